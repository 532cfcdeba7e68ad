// gemm_f64tc against sums in extended precision (a double-double dot product, exact to
// 2^-100), entry by entry.
//
// Bound of an entry, from the split (f64tc.cu): with R the largest magnitude of its row
// of op(A) after k is balanced and C that of its column of op(B), 2^s <= 2.02 R and
// 2^s' <= 2.02 C.  FP64 operands: an entry is rounded 64 bits below 2^s, the slice
// products left out are below 2^-61.1 of 2^s 2^s', so a sum over k is off by at most
// k (2 * 2^-64 + 2^-61.1) 2.02^2 R C < k 2^-58.6 R C.  FP32 operands: seven slices, an
// entry is cut 56 bits below 2^s, six slice products with t = 7 (2^-53.4) are left out:
// k (2 * 2^-56 + 2^-53.3) 2.02^2 R C < k 2^-50.9 R C.  On top the sum is rounded once
// and multiplied and added once: 2^-53 (2 |alpha sum| + |result|).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "dense.cuh"

using namespace hif;

struct Case {
  const char* name;
  int m, n, k, ta, tb, kz, lower, same, kbal, nops;
  double scale_k, scale_r;   // decades of the scales of k and of the rows and columns
  float alpha, beta;
};

// sum of products, as a double-double
struct Sum {
  double hi = 0.0, lo = 0.0;
  void add(double a, double b) {
    const double p = a * b, e = std::fma(a, b, -p);
    const double s = hi + p, z = s - hi;
    lo += (hi - (s - z)) + (p - z) + e;
    hi = s;
  }
};

template <typename S>
static int run(const Case& c, std::mt19937_64& rng) {
  std::normal_distribution<double> nd;
  std::uniform_real_distribution<double> ud(-1, 1);
  const bool same = c.same != 0;
  const int lda = (c.ta ? c.k : c.m) + 3, ldb = same ? lda : (c.tb ? c.n : c.k) + 2, ldc = c.m + 1;
  const size_t na = (size_t)lda * (c.ta ? c.m : c.k), nb = (size_t)ldb * (c.tb ? c.k : c.n), nc = (size_t)ldc * c.n;
  std::vector<GemmOp> ops;
  std::vector<S> A(na * c.nops), B(same ? 1 : nb * c.nops);
  std::vector<double> C(nc * c.nops);
  std::vector<int> e((size_t)c.k * c.nops);
  auto ia = [&](int o, int r, int k) { return na * o + (c.ta ? k + (size_t)r * lda : r + (size_t)k * lda); };
  auto ib = [&](int o, int k, int q) { return nb * o + (c.tb ? q + (size_t)k * ldb : k + (size_t)q * ldb); };
  for (int o = 0; o < c.nops; ++o) {
    GemmOp op{(int64_t)(na * o), same ? (int64_t)(na * o) : (int64_t)(nb * o), (int64_t)(nc * o), c.m, c.n, c.k,
              lda, ldb, ldc, c.ta, c.tb, c.alpha, c.beta, c.lower, c.kz, c.kbal, (int64_t)c.k * o};
    ops.push_back(op);
    std::vector<double> dr(c.m), dq(c.n);
    for (double& v : dr) v = std::pow(10.0, c.scale_r * ud(rng));
    for (double& v : dq) v = std::pow(10.0, c.scale_r * ud(rng));
    for (int k = 0; k < c.k; ++k) {
      // op(A) carries d in k (KB_DOWN) or 1 / d (KB_UP), op(B) the inverse
      const double d = std::pow(10.0, c.scale_k * ud(rng));
      e[(size_t)c.k * o + k] = std::ilogb(d);
      const double sa = c.kbal == KB_NONE || same ? 1.0 : c.kbal == KB_UP ? 1.0 / d : d, sb = 1.0 / sa;
      for (int r = 0; r < c.m; ++r)
        A[ia(o, r, k)] = (S)(c.kz == KZ_A_LOW && k > r ? 0.0 : nd(rng) * sa * dr[r]);
      if (!same)
        for (int q = 0; q < c.n; ++q) {
          const bool zero = (c.kz == KZ_B_UP && k > q) || (c.kz == KZ_B_LOW && k < q);
          B[ib(o, k, q)] = (S)(zero ? 0.0 : nd(rng) * sb * dq[q]);
        }
    }
    for (size_t j = 0; j < nc; ++j) C[nc * o + j] = nd(rng);
  }
  S *dA, *dB;
  double* dC;
  GemmOp* dO;
  int *fl, *de;
  HIF_CUDA_TRY(cudaMalloc(&dA, A.size() * sizeof(S)));
  HIF_CUDA_TRY(cudaMalloc(&dB, B.size() * sizeof(S)));
  HIF_CUDA_TRY(cudaMalloc(&dC, C.size() * 8));
  HIF_CUDA_TRY(cudaMalloc(&dO, ops.size() * sizeof(GemmOp)));
  HIF_CUDA_TRY(cudaMalloc(&fl, sizeof(int) * FLAG_COUNT));
  HIF_CUDA_TRY(cudaMalloc(&de, e.size() * sizeof(int)));
  HIF_CUDA_TRY(cudaMemset(fl, 0xff, sizeof(int) * FLAG_COUNT));
  HIF_CUDA_TRY(cudaMemcpy(dA, A.data(), A.size() * sizeof(S), cudaMemcpyHostToDevice));
  HIF_CUDA_TRY(cudaMemcpy(dB, B.data(), B.size() * sizeof(S), cudaMemcpyHostToDevice));
  HIF_CUDA_TRY(cudaMemcpy(dC, C.data(), C.size() * 8, cudaMemcpyHostToDevice));
  HIF_CUDA_TRY(cudaMemcpy(dO, ops.data(), ops.size() * sizeof(GemmOp), cudaMemcpyHostToDevice));
  HIF_CUDA_TRY(cudaMemcpy(de, e.data(), e.size() * sizeof(int), cudaMemcpyHostToDevice));
  gemm_f64tc<S>(dO, ops.data(), c.nops, dA, same ? dA : dB, dC, fl, 0, "check", de);
  HIF_CUDA_TRY(cudaDeviceSynchronize());
  std::vector<double> R(C.size());
  int flags[FLAG_COUNT];
  HIF_CUDA_TRY(cudaMemcpy(R.data(), dC, R.size() * 8, cudaMemcpyDeviceToHost));
  HIF_CUDA_TRY(cudaMemcpy(flags, fl, sizeof(flags), cudaMemcpyDeviceToHost));
  for (void* p : {(void*)dA, (void*)dB, (void*)dC, (void*)dO, (void*)fl, (void*)de}) cudaFree(p);
  const double unit = sizeof(S) == 8 ? std::ldexp(1.0, -58) / std::pow(2.0, 0.6) : std::ldexp(1.0, -50) / std::pow(2.0, 0.9);
  // by maxima, t_k is not known here: within a factor 2 of none for entries of one scale
  const double slack = c.kbal == KB_MAX && !same ? 4.0 : 1.0;
  int bad = flags[FLAG_TIMEOUT] >= 0;
  double worst = 0, err2 = 0, nrm2 = 0;
  // all entries of small products, 4000 drawn ones of large ones
  const int64_t entries = (int64_t)c.m * c.n;
  const int64_t checks = entries <= 70000 ? entries : 4000;
  for (int o = 0; o < c.nops; ++o)
    for (int64_t t = 0; t < checks; ++t) {
      const int64_t at = checks == entries ? t : (int64_t)(rng() % (uint64_t)entries);
      const int r = (int)(at % c.m), q = (int)(at / c.m);
      if (c.lower && r < q) continue;
      Sum s;
      double ra = 0, cb = 0;   // largest balanced magnitudes
      for (int k = 0; k < c.k; ++k) {
        const double a = (double)A[ia(o, r, k)];
        // A A^T: B is the same array, column q of op(B) is row q of op(A)
        const double b = same ? (double)A[ia(o, q, k)] : (double)B[ib(o, k, q)];
        const int sh = c.kbal == KB_NONE || same || c.kbal == KB_MAX ? 0 : c.kbal == KB_UP ? e[(size_t)c.k * o + k] : -e[(size_t)c.k * o + k];
        ra = std::max(ra, std::fabs(std::ldexp(a, sh)));
        cb = std::max(cb, std::fabs(std::ldexp(b, -sh)));
        s.add(a, b);
      }
      const double al = (double)c.alpha, c0 = c.beta != 0.f ? C[nc * o + r + (size_t)q * ldc] : 0.0;
      const double got = R[nc * o + r + (size_t)q * ldc];
      // got - (c0 + al (hi + lo)), alpha is +-1 here
      const double err = std::fabs(((got - c0) - al * s.hi) - al * s.lo);
      const double bound = std::fabs(al) * c.k * slack * unit * ra * cb +
                           std::ldexp(1.0, -53) * (2.0 * std::fabs(s.hi) + std::fabs(got) + std::fabs(c0));
      worst = std::max(worst, err / bound);
      err2 += err * err;
      nrm2 += s.hi * s.hi;
      if (!(err <= bound)) ++bad;
    }
  std::printf("%s %s: %d of the bound's entries exceeded, worst %.3f of it, error in norm %.1e\n", c.name,
              sizeof(S) == 8 ? "fp64" : "fp32", bad, worst, std::sqrt(err2 / std::max(nrm2, 1e-300)));
  return bad;
}

int main() try {
  std::mt19937_64 rng(20260501);
  const Case cases[] = {
      {"one entry", 1, 1, 1, 0, 0, 0, 0, 0, KB_NONE, 2, 0, 0, 1.f, 0.f},
      {"one tile", 64, 64, 64, 0, 0, 0, 0, 0, KB_NONE, 3, 0, 0, 1.f, 0.f},
      {"ragged", 130, 65, 17, 0, 1, 0, 0, 0, KB_NONE, 2, 0, 2, -1.f, 1.f},
      {"128 k and one more", 129, 63, 129, 1, 0, 0, 0, 0, KB_NONE, 2, 0, 0, 1.f, 0.f},
      {"panel", 200, 64, 64, 0, 1, KZ_B_UP, 0, 0, KB_DOWN, 2, 6, 3, 1.f, 0.f},
      {"X^T", 150, 129, 129, 0, 1, KZ_B_UP, 0, 0, KB_DOWN, 2, 4, 2, 1.f, 0.f},
      {"merge, first", 100, 96, 96, 0, 0, KZ_B_LOW, 0, 0, KB_NONE, 2, 0, 3, 1.f, 0.f},
      {"merge, second", 97, 64, 97, 0, 0, KZ_A_LOW, 0, 0, KB_UP, 2, 6, 0, -1.f, 0.f},
      {"A A^T, 64 k", 200, 200, 64, 0, 1, 0, 1, 1, KB_MAX, 3, 0, 3, -1.f, 1.f},
      {"A A^T, deep", 300, 300, 513, 0, 1, 0, 1, 1, KB_MAX, 2, 0, 3, -1.f, 1.f},
      {"A^T A", 128, 128, 700, 1, 0, 0, 1, 1, KB_MAX, 1, 0, 3, 1.f, 0.f},
      {"by maxima", 300, 257, 200, 1, 0, 0, 0, 0, KB_MAX, 2, 0, 2, -1.f, 1.f},
      {"deep", 256, 250, 2000, 0, 0, 0, 0, 0, KB_NONE, 1, 0, 0, 1.f, 0.f},
      // 0.8 GB of slices each: two launches
      {"more than the work space", 2100, 2048, 12288, 0, 0, 0, 0, 0, KB_NONE, 2, 0, 0, 1.f, 0.f},
  };
  int bad = 0;
  for (const Case& c : cases) bad += run<double>(c, rng);
  for (const Case& c : cases)
    if (c.scale_k == 0.0 && c.k <= 2000) bad += run<float>(c, rng);
  std::printf("%s\n", bad ? "FAILED" : "OK");
  return bad ? 1 : 0;
} catch (const Error& e) {
  std::printf("%s\n", e.msg.c_str());
  return 2;
}
