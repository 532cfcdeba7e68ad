// The two forms of the apply's mat-vecs (gemv.cu): a list short enough for the fine one
// and the same list many times over, which takes the coarse one, have to give every
// column the same bits, in any block of right-hand sides; and both are the product, to
// the rounding of a sum of that length (|y - ref| <= (len + 2) u sum |m x|, u the unit
// roundoff, the reference in long double).
#include <cmath>
#include <cstring>
#include <cstdio>
#include <random>
#include <vector>

#include "dense.cuh"

using namespace hif;

struct Shape {
  int rows, cols, tri, beta;
};

template <typename T>
static int run(std::mt19937_64& rng) {
  std::normal_distribution<double> nd;
  const Shape shapes[] = {{1, 1, 0, 0},    {27, 27, 1, 0},   {64, 64, 1, 1},  {65, 33, 0, 1},   {33, 65, 0, 0},
                          {200, 97, 0, 1}, {343, 343, 1, 0}, {70, 513, 0, 0}, {513, 129, 0, 1}, {129, 129, 1, 1},
                          {700, 640, 0, 0}};
  constexpr int COPIES = 40, COLS = 16;
  int bad = 0;
  for (int trans = 0; trans < 2; ++trans) {
    // one set of operations; copy c of it writes its own part of the work vector
    std::vector<GemvOp> set;
    std::vector<T> M;
    int64_t xs = 0, ys = 0;
    for (const Shape& s : shapes) {
      GemvOp o{};
      o.M = (int64_t)M.size();
      o.rows = s.rows;
      o.cols = s.cols;
      o.ld = s.rows + 1;
      o.tri = s.tri;
      o.alpha = s.beta ? -1.f : 1.f;
      o.beta_one = s.beta;
      o.x = xs;
      o.y = ys;   // from the start of the copy's part
      xs += trans ? s.rows : s.cols;
      ys += trans ? s.cols : s.rows;
      for (int64_t e = 0; e < (int64_t)o.ld * s.cols; ++e) M.push_back((T)nd(rng));
      set.push_back(o);
    }
    const int64_t vs = xs + ys * COPIES;
    std::vector<T> w0((size_t)vs * COLS);
    for (int q = 0; q < COLS; ++q)
      for (int64_t i = 0; i < vs; ++i) w0[(size_t)q * vs + i] = i < xs + ys ? (T)nd(rng) : w0[(size_t)q * vs + xs + (i - xs) % ys];
    T *dM, *dw;
    HIF_CUDA_TRY(cudaMalloc(&dM, M.size() * sizeof(T)));
    HIF_CUDA_TRY(cudaMalloc(&dw, w0.size() * sizeof(T)));
    HIF_CUDA_TRY(cudaMemcpy(dM, M.data(), M.size() * sizeof(T), cudaMemcpyHostToDevice));
    auto apply = [&](int copies, int nrhs) {
      std::vector<GemvOp> ops;
      for (int c = 0; c < copies; ++c)
        for (GemvOp o : set) {
          o.y += xs + c * ys;
          ops.push_back(o);
        }
      std::vector<GemvTask> tasks;
      int cnt[4];
      gemv_plan(ops.data(), (int)ops.size(), trans, tasks, cnt);
      GemvOp* dops;
      GemvTask* dt;
      HIF_CUDA_TRY(cudaMalloc(&dops, ops.size() * sizeof(GemvOp)));
      HIF_CUDA_TRY(cudaMalloc(&dt, tasks.size() * sizeof(GemvTask)));
      HIF_CUDA_TRY(cudaMemcpy(dops, ops.data(), ops.size() * sizeof(GemvOp), cudaMemcpyHostToDevice));
      HIF_CUDA_TRY(cudaMemcpy(dt, tasks.data(), tasks.size() * sizeof(GemvTask), cudaMemcpyHostToDevice));
      HIF_CUDA_TRY(cudaMemcpy(dw, w0.data(), w0.size() * sizeof(T), cudaMemcpyHostToDevice));
      const GemvList<T> list{dops, dt, dM, dw, vs, {cnt[0], cnt[1], cnt[2], cnt[3]}, 0};
      gemv_batched<T>(ops.data(), (int)ops.size(), list, trans, nrhs, 0);
      std::vector<T> w(w0.size());
      HIF_CUDA_TRY(cudaMemcpy(w.data(), dw, w.size() * sizeof(T), cudaMemcpyDeviceToHost));
      cudaFree(dops);
      cudaFree(dt);
      std::printf("%s trans %d, %d columns, %d blocks\n", sizeof(T) == 8 ? "fp64" : "fp32", trans, nrhs, gemv_ctas(cnt));
      return w;
    };
    const std::vector<T> fine = apply(1, 1);
    for (const GemvOp& o : set) {
      const int ny = trans ? o.cols : o.rows;
      for (int i = 0; i < ny; ++i) {
        long double s = 0, ab = 0;
        const int len = trans ? o.rows : o.cols;
        for (int j = 0; j < len; ++j) {
          const int r = trans ? j : i, c = trans ? i : j;
          if (o.tri && c > r) continue;
          const long double p = (long double)M[o.M + r + (int64_t)c * o.ld] * w0[o.x + j];
          s += p;
          ab += std::fabs(p);
        }
        const long double y0 = o.beta_one ? w0[xs + o.y + i] : 0.0L;
        const long double err = std::fabs((long double)fine[xs + o.y + i] - (y0 + (long double)o.alpha * s));
        const double u = sizeof(T) == 8 ? 0x1p-53 : 0x1p-24;
        if (!(err <= (len + 2) * (long double)u * (ab + std::fabs(y0)))) ++bad;
      }
    }
    for (int nrhs : {1, 2, 3, 4, 5, 8, 11, 16}) {
      const std::vector<T> few = apply(1, nrhs), many = apply(COPIES, nrhs);
      for (int q = 0; q < nrhs; ++q)
        for (int64_t i = 0; i < ys; ++i) {
          const T want = few[(size_t)q * vs + xs + i];
          if (q == 0 && std::memcmp(&want, &fine[xs + i], sizeof(T))) ++bad;
          for (int c = 0; c < COPIES; ++c)
            if (std::memcmp(&want, &many[(size_t)q * vs + xs + c * ys + i], sizeof(T))) ++bad;
        }
    }
    cudaFree(dM);
    cudaFree(dw);
  }
  return bad;
}

int main() try {
  std::mt19937_64 rng(20260601);
  const int bad = run<float>(rng) + run<double>(rng);
  std::printf("%d differences\n%s\n", bad, bad ? "FAILED" : "OK");
  return bad ? 1 : 0;
} catch (const Error& e) {
  std::printf("%s\n", e.msg.c_str());
  return 2;
}
