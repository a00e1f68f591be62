// Device self-checks behind qtt_selftest: each kernel family against an
// independent computation on seeded random operands.
#include <cmath>
#include <stdexcept>
#include <string>
#include <utility>
#include <vector>

#include "gemm_tc.cuh"
#include "kernels.cuh"

namespace qtt {

namespace {
struct DBuf {
  double* p = nullptr;
  explicit DBuf(size_t n) {
    if (cudaMalloc(&p, (n + 16) * sizeof(double)) != cudaSuccess) throw std::runtime_error("ENOMEM: selftest");
  }
  ~DBuf() { cudaFree(p); }
};

// FP64 throughput probes.  Every thread runs kChains independent dependency
// chains (enough to hide the pipeline latency) for `iters` rounds; the final
// values are summed into *sink so that nothing is dead code.
constexpr int kChains = 8;

__global__ void __launch_bounds__(256) dfma_rate_kernel(int iters, double a, double b, double* sink) {
  double x[kChains];
#pragma unroll
  for (int c = 0; c < kChains; ++c) x[c] = 1.0 + 1e-3 * (threadIdx.x + c);
  for (int it = 0; it < iters; ++it)
#pragma unroll
    for (int c = 0; c < kChains; ++c) x[c] = fma(x[c], a, b);
  double s = 0.0;
#pragma unroll
  for (int c = 0; c < kChains; ++c) s += x[c];
  if (s == 12345.678) *sink = s;  // never true for the operands used; keeps the chains live
}

// mma.sync.m8n8k4 in FP64 (one warp: D = A B + C, 8 x 8 x 4, 256 FMAs), four
// independent accumulators per warp.
__global__ void __launch_bounds__(256) dmma_rate_kernel(int iters, double a, double b, double* sink) {
  double d[4][2];
#pragma unroll
  for (int c = 0; c < 4; ++c) d[c][0] = d[c][1] = 1e-3 * (threadIdx.x + c);
  const double av = a + 1e-9 * threadIdx.x, bv = b;
  for (int it = 0; it < iters; ++it)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                   : "+d"(d[c][0]), "+d"(d[c][1])
                   : "d"(av), "d"(bv));
  double s = 0.0;
#pragma unroll
  for (int c = 0; c < 4; ++c) s += d[c][0] + d[c][1];
  if (s == 12345.678) *sink = s;
}

std::vector<double> down(const double* d, size_t n) {
  std::vector<double> h(n);
  if (cudaMemcpy(h.data(), d, n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess)
    throw std::runtime_error("CUDA error: selftest copy");
  return h;
}
// The larger of the worst value so far and d, a NaN once there is one (std::fmax would drop it).
double worse(double worst, double d) { return d > worst || std::isnan(d) ? d : worst; }

// Of Q (m x n, row-major): max |Q^T Q - I|, ||Y - Q Q^T Y||_F / ||Y||_F and the
// same of the worst column.
struct QrErrors {
  double orth, resid, worst;
};
QrErrors qr_errors(int m, int n, const std::vector<double>& y, const std::vector<double>& q) {
  QrErrors e{0, 0, 0};
  for (int a = 0; a < n; ++a)
    for (int b = 0; b < n; ++b) {
      double s = 0;
      for (int i = 0; i < m; ++i) s += q[(size_t)i * n + a] * q[(size_t)i * n + b];
      e.orth = worse(e.orth, std::fabs(s - (a == b ? 1.0 : 0.0)));
    }
  double num = 0, den = 0;
  for (int c = 0; c < n; ++c) {
    std::vector<double> coef(n, 0.0);
    double cn = 0, cd = 0;
    for (int a = 0; a < n; ++a)
      for (int i = 0; i < m; ++i) coef[a] += q[(size_t)i * n + a] * y[(size_t)i * n + c];
    for (int i = 0; i < m; ++i) {
      double r = y[(size_t)i * n + c];
      for (int a = 0; a < n; ++a) r -= q[(size_t)i * n + a] * coef[a];
      cn += r * r;
      cd += y[(size_t)i * n + c] * y[(size_t)i * n + c];
    }
    num += cn;
    den += cd;
    if (cd > 0) e.worst = worse(e.worst, std::sqrt(cn / cd));
  }
  e.resid = std::sqrt(num / den);
  return e;
}
}  // namespace

// which = 0: tensor-core GEMM modes against the FP64 GEMM.  For every case
// and mode (BF16X3, TF32, TF32X3, BF16, BF16X6, BF16X10) one value:
// max |C_tc - C_64| / max |C_64|.
// which = 1: QR (FP64, FP32, FP32 + one FP64 Newton-Schulz step): ||Q^T Q - I||_max and
//   ||Q Q^T Y - Y|| / ||Y|| per case and run.
// which = 2: eigensolver (FP64 and FP32): ||G U - U diag(lam)|| / ||G|| and ||U^T U - I||_max.
// which = 3: bias of the tensor-core modes (TF32X3, BF16X3, BF16X6) on positive
// operands, K in {32, 256, 2048}, with and without a one-k-block cap per
// accumulator: (mean, max) of the signed relative error (C_tc - C_64) / C_64.
// which = 7: the CUDA-core GEMMs (FP64, and the small products in FP64 and
// FP32) against a host sum: per case the kind, the terms of a dot product and
// max |C - C_host| / (|alpha| sum |a b| + |beta c0|).
// which = 8: the FP64 eigensolver on a batch of problems of different sizes:
// per problem ||G U - U diag(lam)|| / ||G||, ||U^T U - I||_max and 1 if the
// eigenvalues are not descending, for the leading k columns.
// which = 9: the one-launch tensor-core GEMM against a host sum: per case the
// mode, the terms of a dot product, max and mean of (C - C_host) / (|alpha|
// sum |a b| + |beta c0|); -1 where it does not take the shape.
// which = 12: its two-piece sums on operands whose sums are exact, the second
// piece 2^-30 of the first: per case max |C - C_host|, -1 where it does not
// take the shape.
// which = 15: the one-launch tensor-core GEMM at the limits of K and on graded
// operands: per case the mode, K, the kind (0 Gaussian, 1 graded, 2 graded with
// zeros) and max |C - C_host| / sum |a b| (0 / 0 counts as 0), -1 where it does
// not take the shape.
// which = 13 (no GPU): the QR measures of 1 and 10 on an exact Q, one with a
// NaN and one of NaN: orthonormality, residual, worst column's residual.
std::vector<double> run_selftest(int which) {
  if (which == 13) {
    // Q = the first n columns of I and Y = Q: exact, one NaN in Q, Q all NaN
    const int m = 5, n = 3;
    std::vector<double> q((size_t)m * n, 0.0), v;
    for (int i = 0; i < n; ++i) q[(size_t)i * n + i] = 1.0;
    const std::vector<double> y = q;
    for (int kind = 0; kind < 3; ++kind) {
      if (kind == 1) q[4 * n + 1] = std::nan("");
      if (kind == 2) q.assign(q.size(), std::nan(""));
      const QrErrors e = qr_errors(m, n, y, q);
      v.insert(v.end(), {e.orth, e.resid, e.worst});
    }
    return v;
  }
  cudaStream_t st = nullptr;
  std::vector<double> out;
  int* err = nullptr;
  if (cudaMalloc(&err, 16) != cudaSuccess) throw std::runtime_error("ENOMEM: selftest");
  cudaMemset(err, 0, 16);
  if (which == 0) {
    struct Case {
      int M, N, K, outer, inner;
      bool ta, tb;
      double beta;
    };
    const Case cases[] = {
        {128, 128, 64, 1, 1, false, false, 0.0},  {300, 136, 200, 1, 1, false, false, 0.0},
        {130, 70, 100, 3, 2, true, false, 0.0},  {272, 136, 5000, 1, 1, false, true, 0.0},
        {256, 256, 128, 2, 1, false, false, 0.5}, {136, 160, 272, 1, 1, true, true, 1.0},
        {17, 300, 40, 4, 1, false, false, 0.0}};
    const size_t ws_elems = (size_t)32 << 20;
    DBuf ws(ws_elems);
    size_t pack_bytes = (size_t)256 << 20;
    void* pack = nullptr;
    if (cudaMalloc(&pack, pack_bytes) != cudaSuccess) throw std::runtime_error("ENOMEM: selftest pack");
    unsigned long long seed = 12345;
    for (const Case& c : cases) {
      const long long batch = (long long)c.outer * c.inner;
      const size_t asz = (size_t)c.M * c.K * batch, bsz = (size_t)c.K * c.N * batch, csz = (size_t)c.M * c.N * batch;
      DBuf A(asz), B(bsz), C0(csz), C1(csz);
      fill_gaussian(st, A.p, asz, 1.0, seed++, 1);
      fill_gaussian(st, B.p, bsz, 1.0, seed++, 2);
      MatView av, bv;
      av.p = A.p;
      av.rs = c.ta ? 1 : c.K;
      av.cs = c.ta ? c.M : 1;
      av.si = (long long)c.M * c.K;
      av.so = av.si * c.inner;
      bv.p = B.p;
      bv.rs = c.tb ? 1 : c.N;
      bv.cs = c.tb ? c.K : 1;
      bv.si = (long long)c.K * c.N;
      bv.so = bv.si * c.inner;
      for (int mode = 0; mode < 6; ++mode) {
        fill_gaussian(st, C0.p, csz, 1.0, 777, 3);
        fill_gaussian(st, C1.p, csz, 1.0, 777, 3);
        OutView c0, c1;
        c0.p = C0.p;
        c0.rs = c.N;
        c0.cs = 1;
        c0.si = (long long)c.M * c.N;
        c0.so = c0.si * c.inner;
        c1 = c0;
        c1.p = C1.p;
        gemm_f64(st, c.M, c.N, c.K, c.outer, c.inner, 1.5, av, bv, c.beta, c0, ws.p, ws_elems);
        const int tc_mode[6] = {TC_BF16X3, TC_TF32, TC_TF32X3, TC_BF16, TC_BF16X6, TC_BF16X10};
        if (!gemm_tc(st, tc_mode[mode], c.M, c.N, c.K, c.outer, c.inner, 1.5, av, bv, c.beta, c1, pack, pack_bytes,
                     ws.p, ws_elems, err)) {
          out.push_back(-1.0);
          continue;
        }
        if (cudaStreamSynchronize(st) != cudaSuccess) throw std::runtime_error("CUDA error: selftest gemm");
        std::vector<double> h0 = down(C0.p, csz), h1 = down(C1.p, csz);
        double mx = 0, md = 0;
        for (size_t i = 0; i < csz; ++i) {
          mx = std::fmax(mx, std::fabs(h0[i]));
          md = worse(md, std::fabs(h0[i] - h1[i]));
        }
        out.push_back(md / (mx > 0 ? mx : 1.0));
      }
    }
    cudaFree(pack);
  } else if (which == 1 || which == 10) {
    // which = 1: Gaussian Y.  which = 10, at the edges of the kernels' sizes: kind 0 Gaussian, 1 every
    // third column zero and a repeated one, 2 columns scaled by 10^(-12 .. 12) and rows by 1 or 10^-9
    // (the residual of the worst column).
    const std::vector<std::pair<int, int>> shapes =
        which == 1 ? std::vector<std::pair<int, int>>{{272, 136}, {64, 33}, {256, 256}, {40, 1}, {288, 143},
                                                      {150, 77}, {200, 120}, {96, 2}, {288, 144}, {160, 80},
                                                      {97, 49}, {161, 81}, {144, 72}}
                   : std::vector<std::pair<int, int>>{{1, 1},    {3, 2},    {32, 32},   {33, 17},  {96, 48},
                                                      {49, 49},  {81, 81},  {224, 112}, {225, 112}, {113, 113},
                                                      {129, 65}, {385, 24}, {384, 100}};
    for (auto& sh : shapes)
      for (int kind = 0; kind < (which == 1 ? 1 : 3); ++kind) {
        const int m = sh.first, n = sh.second;
        DBuf Y((size_t)m * n), Q((size_t)m * n), W((size_t)2 * m * n + n + 64), Qf((size_t)m * n),
            G((size_t)8 * n * n);
        fill_gaussian(st, Y.p, (size_t)m * n, 1.0, 99 + m, 5);
        if (cudaStreamSynchronize(st) != cudaSuccess) throw std::runtime_error("CUDA error: selftest qr");
        std::vector<double> y = down(Y.p, (size_t)m * n);
        if (kind > 0) {
          for (int i = 0; i < m; ++i)
            for (int c = 0; c < n; ++c) {
              double& v = y[(size_t)i * n + c];
              if (kind == 1) v = c % 3 == 2 ? 0.0 : c > 0 && c % 3 == 0 ? y[(size_t)i * n + c - 2] : v;
              if (kind == 2) v *= std::pow(10.0, 12 * (c % 3 - 1)) * ((i + c) % 3 == 0 ? 1e-9 : 1.0);
            }
          if (cudaMemcpy(Y.p, y.data(), y.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
            throw std::runtime_error("CUDA error: selftest qr");
        }
        // FP64 QR; float QR; float QR + one FP64 Newton-Schulz step
        for (int run = 0; run < 3; ++run) {
          if (run < 2) {
            qr_thin(st, m, n, Y.p, Q.p, W.p, run == 0 ? 64 : 32, err);
          } else {
            qr_thin(st, m, n, Y.p, Qf.p, W.p, 32, err);
            newton_schulz_step(st, m, n, Qf.p, G.p, Q.p);
          }
          if (cudaStreamSynchronize(st) != cudaSuccess) throw std::runtime_error("CUDA error: selftest qr");
          std::vector<double> q = down(Q.p, (size_t)m * n);
          const QrErrors e = qr_errors(m, n, y, q);
          out.push_back(e.orth);
          out.push_back(which == 1 ? e.resid : e.worst);
        }
      }
  } else if (which == 2) {
    // (size, spectrum): 0 G = X diag(10^(-6 k / n)) X^T (X Gaussian); with Q
    // orthonormal (Gram-Schmidt of a Gaussian X on the host) G = Q diag(w) Q^T
    // for 1: w_k = 10^(-6 k / 20) for k < 20 and 0 beyond (rank 20), 2: w_k =
    // 1/2 for k < 40 (a 40-fold eigenvalue) and 1 + k / n beyond, 3: w_k =
    // 10^(-30 k / n) (graded far below the double precision of the largest)
    const int cases[][2] = {{136, 0}, {64, 0}, {7, 0}, {1, 0}, {200, 0}, {136, 1}, {136, 2}, {136, 3}, {200, 1}, {200, 3}, {520, 0}};
    for (const auto& cs : cases) {
      const int n = cs[0], kind = cs[1];
      std::vector<double> x((size_t)n * n);
      DBuf X((size_t)n * n), G((size_t)n * n), U((size_t)n * n), L(n),
          W((eig_work_bytes(n, 64) > eig_work_bytes(n, 32) ? eig_work_bytes(n, 64) : eig_work_bytes(n, 32)) / 8 + 128);
      fill_gaussian(st, X.p, (size_t)n * n, 1.0, 4242 + n + 1000 * kind, 6);
      if (cudaStreamSynchronize(st) != cudaSuccess) throw std::runtime_error("CUDA error: selftest eig");
      x = down(X.p, (size_t)n * n);
      std::vector<double> w(n);
      for (int k = 0; k < n; ++k)
        w[k] = kind == 0   ? std::pow(10.0, -6.0 * k / n)
               : kind == 1 ? (k < 20 ? std::pow(10.0, -6.0 * k / 20) : 0.0)
               : kind == 2 ? (k < 40 ? 0.5 : 1.0 + (double)k / n)
                           : std::pow(10.0, -30.0 * k / n);
      if (kind != 0) {  // columns of x orthonormal (modified Gram-Schmidt, twice)
        for (int pass = 0; pass < 2; ++pass)
          for (int k = 0; k < n; ++k) {
            for (int j = 0; j < k; ++j) {
              double d = 0;
              for (int i = 0; i < n; ++i) d += x[(size_t)i * n + j] * x[(size_t)i * n + k];
              for (int i = 0; i < n; ++i) x[(size_t)i * n + k] -= d * x[(size_t)i * n + j];
            }
            double nr = 0;
            for (int i = 0; i < n; ++i) nr += x[(size_t)i * n + k] * x[(size_t)i * n + k];
            nr = std::sqrt(nr);
            for (int i = 0; i < n; ++i) x[(size_t)i * n + k] /= nr;
          }
      }
      std::vector<double> g((size_t)n * n, 0.0);
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
          double s = 0;
          for (int k = 0; k < n; ++k) s += x[(size_t)i * n + k] * x[(size_t)j * n + k] * w[k];
          g[(size_t)i * n + j] = s;
        }
      if (cudaMemcpy(G.p, g.data(), g.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
        throw std::runtime_error("CUDA error: selftest eig upload");
      for (int prec : {64, 32}) {
        eig_sym(st, n, n, G.p, U.p, L.p, W.p, prec, err);
        if (cudaStreamSynchronize(st) != cudaSuccess) throw std::runtime_error("CUDA error: selftest eig");
        std::vector<double> u = down(U.p, (size_t)n * n), lam = down(L.p, n);
        double gn = 0, res = 0, orth = 0, order = 0;
        for (double v : g) gn = std::fmax(gn, std::fabs(v));
        for (int c = 0; c < n; ++c) {
          if (c > 0 && lam[c] > lam[c - 1]) order = 1;
          for (int i = 0; i < n; ++i) {
            double s = 0;
            for (int k = 0; k < n; ++k) s += g[(size_t)i * n + k] * u[(size_t)k * n + c];
            res = worse(res, std::fabs(s - lam[c] * u[(size_t)i * n + c]));
          }
          for (int c2 = 0; c2 < n; ++c2) {
            double s = 0;
            for (int k = 0; k < n; ++k) s += u[(size_t)k * n + c] * u[(size_t)k * n + c2];
            orth = worse(orth, std::fabs(s - (c == c2 ? 1.0 : 0.0)));
          }
        }
        out.push_back(res / gn);
        out.push_back(orth);
        out.push_back(order);
      }
    }
  } else if (which == 3) {
    // accumulation bias: positive operands, signed mean of (C_tc - C_64) / C_64
    const size_t ws_elems = (size_t)64 << 20;
    DBuf ws(ws_elems);
    size_t pack_bytes = (size_t)128 << 20;
    void* pack = nullptr;
    if (cudaMalloc(&pack, pack_bytes) != cudaSuccess) throw std::runtime_error("ENOMEM: selftest pack");
    const int Ks[3] = {32, 256, 2048};
    for (int K : Ks) {
      const int M = 256, N = 128;
      DBuf A((size_t)M * K), B((size_t)K * N), C0((size_t)M * N), C1((size_t)M * N);
      fill_gaussian(st, A.p, (size_t)M * K, 1.0, 31 + K, 7);
      fill_gaussian(st, B.p, (size_t)K * N, 1.0, 37 + K, 8);
      std::vector<double> ha = down(A.p, (size_t)M * K), hb = down(B.p, (size_t)K * N);
      for (double& v : ha) v = std::fabs(v);
      for (double& v : hb) v = std::fabs(v);
      cudaMemcpy(A.p, ha.data(), ha.size() * 8, cudaMemcpyHostToDevice);
      cudaMemcpy(B.p, hb.data(), hb.size() * 8, cudaMemcpyHostToDevice);
      MatView av, bv;
      av.p = A.p; av.rs = K; av.cs = 1;
      bv.p = B.p; bv.rs = N; bv.cs = 1;
      OutView c0, c1;
      c0.p = C0.p; c0.rs = N; c0.cs = 1;
      c1 = c0; c1.p = C1.p;
      gemm_f64(st, M, N, K, 1, 1, 1.0, av, bv, 0.0, c0, ws.p, ws_elems);
      const int modes[3] = {TC_TF32X3, TC_BF16X3, TC_BF16X6};
      for (int mode : modes)
        for (int chunk : {0, 1}) {
          if (!gemm_tc(st, mode, M, N, K, 1, 1, 1.0, av, bv, 0.0, c1, pack, pack_bytes, ws.p, ws_elems, err, chunk)) {
            out.push_back(-1.0);
            out.push_back(-1.0);
            continue;
          }
          cudaStreamSynchronize(st);
          std::vector<double> h0 = down(C0.p, (size_t)M * N), h1 = down(C1.p, (size_t)M * N);
          double mean = 0, mx = 0;
          for (size_t i = 0; i < h0.size(); ++i) {
            const double r = (h1[i] - h0[i]) / h0[i];
            mean += r;
            mx = worse(mx, std::fabs(r));
          }
          out.push_back(mean / (double)h0.size());
          out.push_back(mx);
        }
    }
    cudaFree(pack);
  } else if (which == 4) {
    // throughput of the tensor-core GEMM on large square products (the
    // contraction kernel on a shape that fills the GPU), per call including the
    // operand packing: for n in {4096, 8192} and modes (BF16, BF16X3):
    // n, mode, TFLOP/s (2 n^3 per call, mean of 5 timed calls after 2 untimed
    // ones), max relative error of 16 sampled entries against FP64 dot products
    const size_t ws_elems = (size_t)32 << 20;
    DBuf ws(ws_elems);
    for (int n : {4096, 8192}) {
      const size_t sz = (size_t)n * n;  // 8192^2 FP64: 512 MiB per operand
      DBuf A(sz), B(sz), C(sz);
      fill_gaussian(st, A.p, sz, 1.0, 4242 + n, 9);
      fill_gaussian(st, B.p, sz, 1.0, 4343 + n, 10);
      MatView av, bv;
      av.p = A.p; av.rs = n; av.cs = 1;
      bv.p = B.p; bv.rs = n; bv.cs = 1;
      OutView cv;
      cv.p = C.p; cv.rs = n; cv.cs = 1;
      const int modes[2] = {TC_BF16, TC_BF16X3};
      for (int mode : modes) {
        const size_t pack_bytes = tc_workspace_bytes(n, n, n, 1, mode);
        void* pack = nullptr;
        if (cudaMalloc(&pack, pack_bytes) != cudaSuccess) throw std::runtime_error("ENOMEM: selftest pack");
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        bool ok = true;
        for (int it = 0; it < 2 && ok; ++it)
          ok = gemm_tc(st, mode, n, n, n, 1, 1, 1.0, av, bv, 0.0, cv, pack, pack_bytes, ws.p, ws_elems, err);
        float ms = 0.f;
        if (ok) {
          cudaEventRecord(e0, st);
          for (int it = 0; it < 5; ++it)
            gemm_tc(st, mode, n, n, n, 1, 1, 1.0, av, bv, 0.0, cv, pack, pack_bytes, ws.p, ws_elems, err);
          cudaEventRecord(e1, st);
          if (cudaEventSynchronize(e1) != cudaSuccess) throw std::runtime_error("CUDA error: selftest gemm timing");
          cudaEventElapsedTime(&ms, e0, e1);
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        cudaFree(pack);
        double err_max = -1.0;
        if (ok) {  // row i of A, column j of B and C(i, j) only
          err_max = 0.0;
          std::vector<double> ar(n), bc(n);
          for (int q = 0; q < 16; ++q) {
            const size_t i = ((size_t)q * 2654435761u) % n, j = ((size_t)q * 40503u + 7) % n;
            double cij = 0.0;
            if (cudaMemcpy(ar.data(), A.p + i * n, (size_t)n * 8, cudaMemcpyDeviceToHost) != cudaSuccess ||
                cudaMemcpy2D(bc.data(), 8, B.p + j, (size_t)n * 8, 8, n, cudaMemcpyDeviceToHost) != cudaSuccess ||
                cudaMemcpy(&cij, C.p + i * n + j, 8, cudaMemcpyDeviceToHost) != cudaSuccess)
              throw std::runtime_error("CUDA error: selftest gemm sample");
            double ref = 0.0, mag = 0.0;
            for (int k = 0; k < n; ++k) {
              ref += ar[k] * bc[k];
              mag += std::fabs(ar[k] * bc[k]);
            }
            err_max = worse(err_max, std::fabs(cij - ref) / mag);
          }
        }
        out.push_back((double)n);
        out.push_back((double)mode);
        out.push_back(ok && ms > 0.f ? 2.0 * n * (double)n * n * 5.0 / (ms * 1e-3) / 1e12 : -1.0);
        out.push_back(err_max);
      }
    }
  } else if (which == 5) {
    // tensor-core GEMM operands and results for a check on the host in FP64:
    // per case the header (M, N, K, outer, inner, A transposed, B transposed,
    // beta; alpha is 1.5), the operands A, B and the initial C as stored
    // (batch-major, then row-major or, when transposed, column-major), then C
    // after each mode (BF16X3, TF32, TF32X3, BF16, BF16X6, BF16X10; NaN when a mode
    // does not take the shape)
    struct Case {
      int M, N, K, outer, inner;
      bool ta, tb;
      double beta;
    };
    const Case cases[] = {{272, 136, 2176, 1, 1, false, false, 0.0},
                          {4352, 256, 136, 1, 1, false, false, 0.0},
                          {130, 70, 100, 3, 2, true, false, 0.5},
                          {136, 160, 272, 1, 1, true, true, 1.0}};
    const size_t ws_elems = (size_t)32 << 20;
    DBuf ws(ws_elems);
    size_t pack_bytes = (size_t)256 << 20;
    void* pack = nullptr;
    if (cudaMalloc(&pack, pack_bytes) != cudaSuccess) throw std::runtime_error("ENOMEM: selftest pack");
    unsigned long long seed = 24680;
    for (const Case& c : cases) {
      const long long batch = (long long)c.outer * c.inner;
      const size_t asz = (size_t)c.M * c.K * batch, bsz = (size_t)c.K * c.N * batch, csz = (size_t)c.M * c.N * batch;
      DBuf A(asz), B(bsz), C0(csz), C1(csz);
      fill_gaussian(st, A.p, asz, 1.0, seed++, 1);
      fill_gaussian(st, B.p, bsz, 1.0, seed++, 2);
      fill_gaussian(st, C0.p, csz, 1.0, seed++, 3);
      MatView av, bv;
      av.p = A.p;
      av.rs = c.ta ? 1 : c.K;
      av.cs = c.ta ? c.M : 1;
      av.si = (long long)c.M * c.K;
      av.so = av.si * c.inner;
      bv.p = B.p;
      bv.rs = c.tb ? 1 : c.N;
      bv.cs = c.tb ? c.K : 1;
      bv.si = (long long)c.K * c.N;
      bv.so = bv.si * c.inner;
      OutView cv;
      cv.p = C1.p;
      cv.rs = c.N;
      cv.cs = 1;
      cv.si = (long long)c.M * c.N;
      cv.so = cv.si * c.inner;
      const double hdr[8] = {(double)c.M, (double)c.N, (double)c.K, (double)c.outer, (double)c.inner,
                             c.ta ? 1.0 : 0.0, c.tb ? 1.0 : 0.0, c.beta};
      out.insert(out.end(), hdr, hdr + 8);
      for (const DBuf* d : {&A, &B, &C0}) {
        const std::vector<double> h = down(d->p, d == &A ? asz : d == &B ? bsz : csz);
        out.insert(out.end(), h.begin(), h.end());
      }
      const int tc_mode[6] = {TC_BF16X3, TC_TF32, TC_TF32X3, TC_BF16, TC_BF16X6, TC_BF16X10};
      for (int mode = 0; mode < 6; ++mode) {
        if (cudaMemcpy(C1.p, C0.p, csz * sizeof(double), cudaMemcpyDeviceToDevice) != cudaSuccess)
          throw std::runtime_error("CUDA error: selftest copy");
        if (!gemm_tc(st, tc_mode[mode], c.M, c.N, c.K, c.outer, c.inner, 1.5, av, bv, c.beta, cv, pack, pack_bytes,
                     ws.p, ws_elems, err)) {
          out.insert(out.end(), csz, std::nan(""));
          continue;
        }
        if (cudaStreamSynchronize(st) != cudaSuccess) throw std::runtime_error("CUDA error: selftest gemm");
        const std::vector<double> h = down(C1.p, csz);
        out.insert(out.end(), h.begin(), h.end());
      }
    }
    cudaFree(pack);
  } else if (which == 6) {
    // FP64 arithmetic throughput of the whole GPU: DFMA (CUDA cores) and
    // mma.sync m8n8k4 f64; per probe TFLOP/s (2 flops per FMA) of the best of
    // three timed launches after one untimed one, then the SM count and the
    // number of blocks launched
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    DBuf sink(1);
    const int blocks = sms * 8, threads = 256, iters = 4096;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    for (int probe = 0; probe < 2; ++probe) {
      float best = 1e30f;
      for (int rep = 0; rep < 4; ++rep) {
        cudaEventRecord(e0, st);
        if (probe == 0)
          dfma_rate_kernel<<<blocks, threads, 0, st>>>(iters, 0.999999, 1e-7, sink.p);
        else
          dmma_rate_kernel<<<blocks, threads, 0, st>>>(iters, 0.999999, 1e-7, sink.p);
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) throw std::runtime_error("CUDA error: FP64 rate probe");
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0 && ms < best) best = ms;
      }
      const double fma_per_thread =
          probe == 0 ? (double)iters * kChains : (double)iters * 4 * 256.0 / 32.0;  // 256 FMAs per warp-MMA
      const double flops = 2.0 * fma_per_thread * threads * (double)blocks;
      out.push_back(flops / (best * 1e-3) / 1e12);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    out.push_back((double)sms);
    out.push_back((double)blocks);
  } else if (which == 7) {
    struct Case {
      int kind;  // 0: gemm_f64, 1: small products in FP64, 2: in FP32
      int M, N, K, outer, inner, pieces;
      bool ta, tb, shared_a;  // shared_a: A does not depend on the outer index
      double alpha, beta;
      bool ws;
    };
    const Case cases[] = {
        {0, 1, 1, 1, 1, 1, 1, false, false, false, 1.0, 0.0, false},
        {0, 40, 40, 80, 1, 1, 1, false, true, false, 1.0, 0.0, false},
        {0, 136, 136, 272, 1, 1, 1, true, false, false, 1.0, 0.0, false},
        {0, 33, 73, 31, 3, 2, 1, false, false, false, -1.5, 0.5, false},
        {0, 272, 136, 4000, 1, 1, 1, false, false, false, 1.0, 1.0, true},
        {0, 5, 7, 33, 1, 4, 1, true, true, false, 1.0, 0.0, true},
        {0, 2049, 65, 9, 1, 1, 1, false, false, false, 1.0, 0.0, false},
        {0, 77, 161, 145, 1, 2, 1, true, true, false, 2.0, 0.0, true},
        {1, 1, 1, 1, 1, 1, 1, false, false, true, 1.0, 0.0, false},
        {1, 26, 40, 26, 32, 1, 4, false, false, true, 1.0, 0.0, false},
        {1, 32, 33, 64, 5, 2, 2, false, false, true, 0.5, 2.0, false},
        {1, 8, 31, 7, 3, 2, 1, true, false, false, 1.0, 0.0, false},
        {1, 32, 200, 64, 7, 1, 4, false, true, true, 1.0, 0.0, false},
        {2, 1, 1, 1, 1, 1, 1, false, false, true, 1.0, 0.0, false},
        {2, 26, 136, 26, 128, 1, 4, false, false, true, 1.0, 0.0, false},
        {2, 9, 17, 63, 2, 3, 2, true, false, true, 1.5, 1.0, false},
        {2, 32, 300, 64, 40, 1, 1, false, false, false, 1.0, 0.0, false}};
    const size_t ws_elems = (size_t)4 << 20;
    DBuf ws(ws_elems);
    unsigned long long seed = 4242;
    for (const Case& c : cases) {
      const long long batch = (long long)c.outer * c.inner;
      const size_t am = (size_t)c.M * c.K, bm = (size_t)c.K * c.N, cm = (size_t)c.M * c.N;
      const long long na = (c.shared_a ? c.inner : batch) * c.pieces, nb = batch * c.pieces;
      DBuf A(am * na), B(bm * nb), C0(cm * batch);
      fill_gaussian(st, A.p, am * na, 1.0, seed++, 1);
      fill_gaussian(st, B.p, bm * nb, 1.0, seed++, 2);
      fill_gaussian(st, C0.p, cm * batch, 1.0, seed++, 3);
      const std::vector<double> ha = down(A.p, am * na), hb = down(B.p, bm * nb), hc = down(C0.p, cm * batch);
      MatView av, bv;
      OutView cv;
      av.p = A.p;
      av.rs = c.ta ? 1 : c.K;
      av.cs = c.ta ? c.M : 1;
      av.si = (long long)am * c.pieces;
      av.so = c.shared_a ? 0 : av.si * c.inner;
      bv.p = B.p;
      bv.rs = c.tb ? 1 : c.N;
      bv.cs = c.tb ? c.K : 1;
      bv.si = (long long)bm * c.pieces;
      bv.so = bv.si * c.inner;
      cv.p = C0.p;
      cv.rs = c.N;
      cv.cs = 1;
      cv.si = (long long)cm;
      cv.so = cv.si * c.inner;
      SumPieces P;
      P.n = c.pieces;
      P.a = (long long)am;
      P.b0 = (long long)bm;
      P.b1 = 2 * (long long)bm;
      if (c.kind == 0)
        gemm_f64(st, c.M, c.N, c.K, c.outer, c.inner, c.alpha, av, bv, c.beta, cv, c.ws ? ws.p : nullptr,
                 c.ws ? ws_elems : 0);
      else
        small_gemm_sum(st, c.kind == 2, c.M, c.N, c.K, c.outer, c.inner, c.alpha, av, bv, c.beta, cv, P);
      const std::vector<double> got = down(C0.p, cm * batch);
      double worst = 0.0;
      for (long long b = 0; b < batch; ++b)
        for (int m = 0; m < c.M; ++m)
          for (int n = 0; n < c.N; ++n) {
            double v = 0.0, mag = 0.0, lost = 0.0;  // compensated sum
            for (int p = 0; p < c.pieces; ++p) {
              const double* a = ha.data() + ((c.shared_a ? b % c.inner : b) * c.pieces + p) * am;
              const double* w = hb.data() + (b * c.pieces + p) * bm;
              for (int k = 0; k < c.K; ++k) {
                const double x = a[c.ta ? (size_t)k * c.M + m : (size_t)m * c.K + k];
                const double y = w[c.tb ? (size_t)n * c.K + k : (size_t)k * c.N + n];
                const double t = x * y - lost, s = v + t;
                lost = (s - v) - t;
                v = s;
                mag += std::fabs(x * y);
              }
            }
            const size_t e = (size_t)b * cm + (size_t)m * c.N + n;
            const double ref = c.alpha * v + c.beta * hc[e];
            const double scale = std::fabs(c.alpha) * mag + std::fabs(c.beta * hc[e]);
            const double d = std::fabs(got[e] - ref) / scale;
            worst = worse(worst, d);
          }
      out.push_back((double)c.kind);
      out.push_back((double)c.K * c.pieces);
      out.push_back(worst);
    }
  } else if (which == 8 || which == 11) {
    // 8: sizes at the edges of the leaves (12) and of the levels.  11: batches at
    // the edges of the back-transform's variants.  Every second problem of rank
    // n / 3 (equal poles and negligible z in its merges).
    std::vector<std::vector<int>> batches = {{136, 1, 2, 12, 13, 24, 25, 40, 49, 72, 96, 97, 104, 193}};
    if (which == 11) batches = {{64, 33, 3}, {96, 65, 2, 1}, {160, 97, 145}, {161, 5}};
    for (const std::vector<int>& sizes : batches) {
      const int np = (int)sizes.size();
      std::vector<std::vector<double>> gs(np);
      std::vector<EigProblem> probs(np);
      size_t total = 0;
      for (int n : sizes) total += 3 * (size_t)n * n + n + eig_work_bytes(n, 64) / 8 + 96;
      DBuf mem(total), dev(np * sizeof(EigProblem) / 8 + 8);
      double* p = mem.p;
      int nmax = 0, kmax = 0;
      for (int t = 0; t < np; ++t) {
        const int n = sizes[t];
        EigProblem& P = probs[t];
        P.n = n;
        P.k = t % 3 == 0 ? n : n / 2 + 1;
        double* X = p;
        double* G = X + (size_t)n * n;
        P.G = G;
        P.U = G + (size_t)n * n;
        P.lam = P.U + (size_t)n * n;
        P.work = (unsigned char*)(P.lam + n);
        P.work = (unsigned char*)(((uintptr_t)P.work + 255) & ~(uintptr_t)255);
        p = (double*)(((uintptr_t)P.work + eig_work_bytes(n, 64) + 255) & ~(uintptr_t)255);
        nmax = n > nmax ? n : nmax;
        kmax = P.k > kmax ? P.k : kmax;
        fill_gaussian(st, X, (size_t)n * n, 1.0, 555 + t, 6);
        const std::vector<double> x = down(X, (size_t)n * n);
        std::vector<double>& g = gs[t];
        g.assign((size_t)n * n, 0.0);
        for (int i = 0; i < n; ++i)
          for (int j = 0; j <= i; ++j) {
            double s = 0;
            for (int k = 0; k < n; ++k)
              s += x[(size_t)i * n + k] * x[(size_t)j * n + k] *
                   (t % 2 ? (3 * k < n ? 1.0 : 0.0) : std::pow(10.0, -6.0 * k / n));
            g[(size_t)i * n + j] = g[(size_t)j * n + i] = s;
          }
        if (cudaMemcpy(G, g.data(), g.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
          throw std::runtime_error("CUDA error: selftest eig upload");
      }
      if (cudaMemcpy(dev.p, probs.data(), np * sizeof(EigProblem), cudaMemcpyHostToDevice) != cudaSuccess)
        throw std::runtime_error("CUDA error: selftest eig upload");
      eig_sym_batched(st, (const EigProblem*)dev.p, np, nmax, kmax, 64, err);
      if (cudaStreamSynchronize(st) != cudaSuccess) throw std::runtime_error("CUDA error: selftest eig");
      for (int t = 0; t < np; ++t) {
        const int n = probs[t].n, k = probs[t].k;
        const std::vector<double> u = down(probs[t].U, (size_t)n * k), lam = down(probs[t].lam, n);
        double gn = 0, res = 0, orth = 0, order = 0;
        for (double v : gs[t]) gn = std::fmax(gn, std::fabs(v));
        for (int c = 1; c < n; ++c)
          if (lam[c] > lam[c - 1]) order = 1;
        for (int c = 0; c < k; ++c) {
          for (int i = 0; i < n; ++i) {
            double s = 0;
            for (int q = 0; q < n; ++q) s += gs[t][(size_t)i * n + q] * u[(size_t)q * k + c];
            const double d = std::fabs(s - lam[c] * u[(size_t)i * k + c]);
            res = worse(res, d);
          }
          for (int c2 = 0; c2 < k; ++c2) {
            double s = 0;
            for (int q = 0; q < n; ++q) s += u[(size_t)q * k + c] * u[(size_t)q * k + c2];
            const double d = std::fabs(s - (c == c2 ? 1.0 : 0.0));
            orth = worse(orth, d);
          }
        }
        out.push_back(res / gn);
        out.push_back(orth);
        out.push_back(order);
      }
    }
  } else if (which == 9) {
    struct Case {
      int mode, M, N, K, outer, inner, pieces;
      bool ta, tb, sa, sb;  // transposed operands; operands that do not depend on the outer index
      double alpha, beta;
      bool flip_c;  // C column-major
    };
    const Case cases[] = {
        // rows and columns inside one tile, over tile edges, ragged K; every layout of the rows
        {TC_TF32X3, 128, 144, 32, 1, 1, 1, false, false, false, false, 1.0, 0.0, false},
        {TC_TF32X3, 300, 136, 136, 1, 2, 1, false, true, false, true, 1.0, 0.0, false},
        {TC_TF32X3, 77, 85, 77, 9, 2, 1, false, false, true, false, 1.0, 0.0, false},
        {TC_TF32X3, 128, 136, 77, 5, 1, 2, false, false, true, false, 1.0, 0.0, false},
        {TC_TF32X3, 272, 136, 3000, 1, 1, 1, false, false, false, false, 1.0, 0.0, false},
        {TC_TF32X3, 1, 33, 65, 1, 1, 1, true, true, false, false, -1.0, 0.5, true},
        {TC_BF16X6, 136, 700, 272, 1, 1, 1, true, false, false, false, 1.0, 0.0, false},
        {TC_BF16X6, 650, 256, 128, 1, 1, 1, false, false, false, false, 0.5, 0.0, false},
        {TC_BF16X6, 77, 77, 77, 12, 2, 1, true, false, true, false, 1.0, 0.0, false},
        {TC_BF16X6, 45, 37, 340, 3, 1, 1, false, true, false, true, 1.0, 1.0, true},
        {TC_BF16X10, 136, 300, 272, 1, 1, 1, true, false, false, false, 1.0, 0.0, false},
        {TC_BF16X10, 400, 256, 77, 1, 1, 1, false, false, false, false, -1.0, 0.0, false},
        {TC_BF16X10, 33, 40, 65, 7, 2, 1, false, false, true, false, 1.5, 1.0, false},
        {TC_BF16X10, 130, 16, 9, 1, 3, 1, true, true, false, false, 1.0, 0.0, true},
        {TC_BF16X10, 400, 500, 64, 1, 1, 1, false, false, false, false, 1.0, 0.0, false}};
    const size_t ws_elems = (size_t)8 << 20;
    DBuf ws(ws_elems);
    unsigned long long seed = 99;
    for (const Case& c : cases) {
      const long long batch = (long long)c.outer * c.inner;
      const size_t am = (size_t)c.M * c.K, bm = (size_t)c.K * c.N, cm = (size_t)c.M * c.N;
      const long long na = (c.sa ? c.inner : batch) * c.pieces, nb = (c.sb ? c.inner : batch) * c.pieces;
      DBuf A(am * na), B(bm * nb), C0(cm * batch);
      fill_gaussian(st, A.p, am * na, 1.0, seed++, 1);
      fill_gaussian(st, B.p, bm * nb, 1.0, seed++, 2);
      fill_gaussian(st, C0.p, cm * batch, 1.0, seed++, 3);
      const std::vector<double> ha = down(A.p, am * na), hb = down(B.p, bm * nb), hc = down(C0.p, cm * batch);
      MatView av, bv;
      OutView cv;
      av.p = A.p;
      av.rs = c.ta ? 1 : c.K;
      av.cs = c.ta ? c.M : 1;
      av.si = (long long)am * c.pieces;
      av.so = c.sa ? 0 : av.si * c.inner;
      bv.p = B.p;
      bv.rs = c.tb ? 1 : c.N;
      bv.cs = c.tb ? c.K : 1;
      bv.si = (long long)bm * c.pieces;
      bv.so = c.sb ? 0 : bv.si * c.inner;
      cv.p = C0.p;
      cv.rs = c.flip_c ? 1 : c.N;
      cv.cs = c.flip_c ? c.M : 1;
      cv.si = (long long)cm;
      cv.so = cv.si * c.inner;
      SumPieces P;
      P.n = c.pieces;
      P.a = (long long)am;
      P.b0 = (long long)bm;
      out.push_back((double)c.mode);
      out.push_back((double)c.K * c.pieces);
      if (!gemm_fused(st, c.mode, c.M, c.N, c.K, c.outer, c.inner, c.alpha, av, bv, c.beta, cv, P, ws.p, ws_elems, err)) {
        out.push_back(-1.0);
        out.push_back(0.0);
        continue;
      }
      const std::vector<double> got = down(C0.p, cm * batch);
      double worst = 0.0, mean = 0.0;
      for (long long b = 0; b < batch; ++b)
        for (int m = 0; m < c.M; ++m)
          for (int n = 0; n < c.N; ++n) {
            double v = 0.0, mag = 0.0;
            for (int p = 0; p < c.pieces; ++p) {
              const double* a = ha.data() + ((c.sa ? b % c.inner : b) * c.pieces + p) * am;
              const double* w = hb.data() + ((c.sb ? b % c.inner : b) * c.pieces + p) * bm;
              for (int k = 0; k < c.K; ++k) {
                const double t = a[c.ta ? (size_t)k * c.M + m : (size_t)m * c.K + k] *
                                 w[c.tb ? (size_t)n * c.K + k : (size_t)k * c.N + n];
                v += t;
                mag += std::fabs(t);
              }
            }
            const size_t e = (size_t)b * cm + (c.flip_c ? (size_t)n * c.M + m : (size_t)m * c.N + n);
            const double d = (got[e] - c.alpha * v - c.beta * hc[e]) / (std::fabs(c.alpha) * mag + std::fabs(c.beta * hc[e]));
            worst = worse(worst, std::fabs(d));
            mean += d / ((double)cm * batch);
          }
      out.push_back(worst);
      out.push_back(mean);
    }
  } else if (which == 12) {
    // Whole numbers of at most 4 in magnitude: products and sums of up to 400
    // terms are exact in TF32 and FP32, and so is their FP64 sum with 2^-30 of
    // the same; an FP32 sum of the two pieces keeps none of the second.
    struct Case {
      int M, N, K, outer, inner;
      double alpha, beta;
    };
    const Case cases[] = {{128, 136, 77, 5, 1, 1.0, 0.0}, {300, 144, 32, 1, 1, 1.0, 0.0}, {40, 34, 130, 3, 2, -1.0, 1.0}};
    unsigned int lcg = 1u;
    auto whole = [&](std::vector<double>& v) {
      for (double& x : v) {
        lcg = lcg * 1664525u + 1013904223u;
        x = (double)((int)(lcg >> 24) % 9 - 4);
      }
    };
    for (const Case& c : cases) {
      // A [inner][piece][M][K] (no outer index), B [outer][inner][piece][K][N]
      const long long batch = (long long)c.outer * c.inner;
      const size_t am = (size_t)c.M * c.K, bm = (size_t)c.K * c.N, cm = (size_t)c.M * c.N;
      std::vector<double> ha(am * 2 * c.inner), hb(bm * 2 * batch), hc(cm * batch);
      whole(ha);
      whole(hb);
      whole(hc);
      for (long long b = 0; b < batch; ++b)
        for (size_t e = 0; e < bm; ++e) hb[(2 * b + 1) * bm + e] *= std::ldexp(1.0, -30);
      DBuf A(ha.size()), B(hb.size()), C0(hc.size());
      if (cudaMemcpy(A.p, ha.data(), ha.size() * 8, cudaMemcpyHostToDevice) != cudaSuccess ||
          cudaMemcpy(B.p, hb.data(), hb.size() * 8, cudaMemcpyHostToDevice) != cudaSuccess ||
          cudaMemcpy(C0.p, hc.data(), hc.size() * 8, cudaMemcpyHostToDevice) != cudaSuccess)
        throw std::runtime_error("CUDA error: selftest upload");
      MatView av, bv;
      OutView cv;
      av.p = A.p;
      av.rs = c.K;
      av.cs = 1;
      av.si = 2 * (long long)am;
      av.so = 0;
      bv.p = B.p;
      bv.rs = c.N;
      bv.cs = 1;
      bv.si = 2 * (long long)bm;
      bv.so = bv.si * c.inner;
      cv.p = C0.p;
      cv.rs = c.N;
      cv.cs = 1;
      cv.si = (long long)cm;
      cv.so = cv.si * c.inner;
      SumPieces P;
      P.n = 2;
      P.a = (long long)am;
      P.b0 = (long long)bm;
      if (!gemm_fused(st, TC_TF32X3, c.M, c.N, c.K, c.outer, c.inner, c.alpha, av, bv, c.beta, cv, P, nullptr, 0, err)) {
        out.push_back(-1.0);
        continue;
      }
      const std::vector<double> got = down(C0.p, hc.size());
      double worst = 0.0;
      for (long long b = 0; b < batch; ++b)
        for (int m = 0; m < c.M; ++m)
          for (int n = 0; n < c.N; ++n) {
            double v = 0.0;
            for (int p = 0; p < 2; ++p)
              for (int k = 0; k < c.K; ++k)
                v += ha[((b % c.inner) * 2 + p) * am + (size_t)m * c.K + k] * hb[(b * 2 + p) * bm + (size_t)k * c.N + n];
            const size_t e = (size_t)b * cm + (size_t)m * c.N + n;
            const double d = std::fabs(got[e] - (c.alpha * v + c.beta * hc[e]));
            worst = worse(worst, d);
          }
      out.push_back(worst);
    }
  } else if (which == 15) {
    struct Case {
      int mode, M, N, K;
      bool ta, tb;
      int kind;
    };
    // the largest K of the exact-slice modes and one more; both layouts of either operand
    const Case cases[] = {
        {TC_BF16X10, 150, 136, 448, false, false, 0}, {TC_BF16X10, 150, 70, 449, false, false, 0},
        {TC_BF16X10, 150, 70, 300, true, false, 1},   {TC_BF16X10, 131, 136, 300, false, true, 2},
        {TC_BF16X6, 150, 144, 352, false, false, 0},  {TC_BF16X6, 150, 144, 353, false, false, 0},
        {TC_BF16X6, 150, 70, 330, true, false, 1},    {TC_BF16X6, 131, 140, 330, false, true, 2},
        {TC_TF32X3, 150, 144, 330, false, false, 1},  {TC_TF32X3, 131, 140, 330, true, true, 2}};
    unsigned long long seed = 1357;
    for (const Case& c : cases) {
      const int M = c.M, N = c.N, K = c.K;
      const size_t am = (size_t)M * K, bm = (size_t)K * N, cm = (size_t)M * N;
      DBuf A(am), B(bm), C0(cm);
      fill_gaussian(st, A.p, am, 1.0, seed++, 1);
      fill_gaussian(st, B.p, bm, 1.0, seed++, 2);
      std::vector<double> ha = down(A.p, am), hb = down(B.p, bm);
      auto a = [&](int m, int k) -> double& { return ha[c.ta ? (size_t)k * M + m : (size_t)m * K + k]; };
      auto b = [&](int k, int n) -> double& { return hb[c.tb ? (size_t)n * K + k : (size_t)k * N + n]; };
      if (c.kind > 0) {
        // column k of A times 10^(-12, 0, 12), row k of B by the inverse; rows of A
        // and columns of B over decades; entries 10^-8 and 10^-30 of their neighbours
        for (int k = 0; k < K; ++k) {
          const double g = std::pow(10.0, 12 * (k % 3 - 1));
          for (int m = 0; m < M; ++m)
            a(m, k) *= g * std::pow(10.0, 6 * (m % 5 - 2)) * ((m + k) % 7 == 0 ? 1e-8 : (m + k) % 7 == 1 ? 1e-30 : 1.0);
          for (int n = 0; n < N; ++n) b(k, n) *= std::pow(10.0, 5 * (n % 3 - 1)) / g;
        }
      }
      if (c.kind == 2) {
        // zero rows and columns; K indices that are zero in A, in B (large in the other operand) and in both
        for (int k = 0; k < K; ++k)
          for (int m = 0; m < M; ++m)
            if (m % 41 == 3 || k % 29 == 5 || k % 29 == 7) a(m, k) = 0.0;
            else if (k % 29 == 6) a(m, k) = 1e9 * (1.0 + m % 3);
        for (int k = 0; k < K; ++k)
          for (int n = 0; n < N; ++n)
            if (n % 37 == 2 || k % 29 == 6 || k % 29 == 7) b(k, n) = 0.0;
            else if (k % 29 == 5) b(k, n) = 1e9 * (1.0 + n % 3);
      }
      if (cudaMemcpy(A.p, ha.data(), am * 8, cudaMemcpyHostToDevice) != cudaSuccess ||
          cudaMemcpy(B.p, hb.data(), bm * 8, cudaMemcpyHostToDevice) != cudaSuccess)
        throw std::runtime_error("CUDA error: selftest upload");
      MatView av, bv;
      OutView cv;
      av.p = A.p;
      av.rs = c.ta ? 1 : K;
      av.cs = c.ta ? M : 1;
      bv.p = B.p;
      bv.rs = c.tb ? 1 : N;
      bv.cs = c.tb ? K : 1;
      cv.p = C0.p;
      cv.rs = N;
      cv.cs = 1;
      out.insert(out.end(), {(double)c.mode, (double)K, (double)c.kind});
      if (!gemm_fused(st, c.mode, M, N, K, 1, 1, 1.0, av, bv, 0.0, cv, SumPieces{}, nullptr, 0, err)) {
        out.push_back(-1.0);
        continue;
      }
      const std::vector<double> got = down(C0.p, cm);
      double worst = 0.0;
      for (int m = 0; m < M; ++m)
        for (int n = 0; n < N; ++n) {
          double v = 0.0, mag = 0.0;
          for (int k = 0; k < K; ++k) {
            const double t = a(m, k) * b(k, n);
            v += t;
            mag += std::fabs(t);
          }
          const double d = std::fabs(got[(size_t)m * N + n] - v);
          worst = worse(worst, d == 0.0 ? 0.0 : d / mag);
        }
      out.push_back(worst);
    }
  } else {
    cudaFree(err);
    throw std::runtime_error("EINVAL: unknown selftest");
  }
  int herr[4] = {0, 0, 0, 0};
  cudaMemcpy(herr, err, 16, cudaMemcpyDeviceToHost);
  cudaFree(err);
  if (cudaGetLastError() != cudaSuccess) throw std::runtime_error("CUDA error: selftest launch");
  out.push_back((double)herr[0]);
  return out;
}

}  // namespace qtt
