// Vector kernels: gathers and scatters of the apply sweeps (deterministic, no
// atomics), the seven-point residual in double, dot products and updates of
// the preconditioned conjugate gradients.
#include <algorithm>

#include "solve.cuh"

namespace hif {

namespace {

constexpr int VT = 256;
constexpr int PCG_BLOCKS = 1024;   // blocks per column, at most

template <typename T>
__global__ void k_gather(const int32_t* __restrict__ idx, int64_t cnt, const T* __restrict__ y,
                         int64_t ys, T* work, int64_t vs, int64_t voff, int nrhs) {
  const int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x;
  if (i >= cnt) return;
  const int64_t g = idx[i];
  for (int q = 0; q < nrhs; ++q) work[q * vs + voff + i] = y[q * ys + g];
}

template <typename T>
__global__ void k_set(const int32_t* __restrict__ gi, const int32_t* __restrict__ pos, int64_t cnt,
                      T* y, int64_t ys, const T* __restrict__ work, int64_t vs, int nrhs) {
  const int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x;
  if (i >= cnt) return;
  const int64_t g = gi[i], p = pos[i];
  for (int q = 0; q < nrhs; ++q) y[q * ys + g] = work[q * vs + p];
}

template <typename T>
__global__ void k_acc(const int32_t* __restrict__ tgt, const int64_t* __restrict__ ptr,
                      const int32_t* __restrict__ src, int64_t ntgt, T* y, int64_t ys,
                      const T* __restrict__ work, int64_t vs, int nrhs) {
  const int64_t t = (int64_t)blockIdx.x * VT + threadIdx.x;
  if (t >= ntgt) return;
  const int64_t g = tgt[t];
  for (int q = 0; q < nrhs; ++q) {
    T s = T(0);
    for (int64_t e = ptr[t]; e < ptr[t + 1]; ++e) s += work[q * vs + src[e]];
    y[q * ys + g] -= s;
  }
}

template <typename T>
__global__ void k_cin(const double* __restrict__ x, T* y, int64_t cnt) {
  const int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x;
  if (i < cnt) y[i] = (T)x[i];
}

template <typename T>
__global__ void k_cout(const T* __restrict__ y, double* x, int64_t cnt) {
  const int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x;
  if (i < cnt) x[i] = (double)y[i];
}

// The row of the seven-point operator at point j.  Dirichlet: neighbours outside
// the grid are absent; periodic: index arithmetic wraps around every dimension.
struct StencilRow {
  double diag, c[6];   // couplings to +x, -x, +y, -y, +z, -z
  int off[6];          // neighbour offsets, 0: absent
};
__device__ __forceinline__ StencilRow stencil_row(const double* __restrict__ cpl,
                                                  const double* __restrict__ diag, int n,
                                                  int periodic, int64_t j) {
  const int nn = n * n;
  const int64_t N = (int64_t)nn * n;
  const int x2 = (int)(j / nn), rem = (int)(j - (int64_t)x2 * nn), x1 = rem / n, x0 = rem - x1 * n;
  const int x[3] = {x0, x1, x2}, step[3] = {1, n, nn};
  StencilRow r;
  r.diag = diag[j];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int wrap = periodic ? (n - 1) * step[d] : 0;
    r.off[2 * d] = x[d] + 1 < n ? step[d] : -wrap;
    r.off[2 * d + 1] = x[d] > 0 ? -step[d] : wrap;
    r.c[2 * d] = r.off[2 * d] ? cpl[d * N + j] : 0.0;
    r.c[2 * d + 1] = r.off[2 * d + 1] ? cpl[d * N + j + r.off[2 * d + 1]] : 0.0;
  }
  return r;
}
__device__ __forceinline__ double stencil_apply(const StencilRow& r, const double* __restrict__ u,
                                                int64_t j) {
  double s = r.diag * u[j];
#pragma unroll
  for (int i = 0; i < 6; ++i)
    if (r.off[i]) s -= r.c[i] * u[j + r.off[i]];
  return s;
}

// r = f - A u, one point of every column per thread.  Bound by the FP64 unit, 8
// operations per point and column (128^3, 3 columns: 95 us of 115; HBM 32 us).
__global__ void __launch_bounds__(VT) k_residual(const double* __restrict__ cpl,
                                                 const double* __restrict__ diag, int n,
                                                 int periodic, const double* __restrict__ f,
                                                 const double* __restrict__ u, double* out,
                                                 int nrhs) {
  const int64_t N = (int64_t)n * n * n;
  const int64_t j = (int64_t)blockIdx.x * VT + threadIdx.x;
  if (j >= N) return;
  const StencilRow row = stencil_row(cpl, diag, n, periodic, j);
  for (int q = 0; q < nrhs; ++q)
    out[q * N + j] = f[q * N + j] - stencil_apply(row, u + q * N, j);
}

// ---- conjugate gradients ---------------------------------------------------------
// Bound by HBM and, for the operator and the dot products, by the FP64 unit; on
// small grids by the launches and host waits.  So each pass over the vectors
// does all that its operands allow, its sums end in a one-block kernel per
// column that forms the next coefficient, and nothing is copied: an iteration
// is seven launches and one wait (it was eleven, three copies and three waits).
// Column c is blockIdx.y; sums are added in a fixed order.

// sum over the block, valid in thread 0
__device__ __forceinline__ double block_sum(double s) {
  __shared__ double red[VT / 32];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __syncthreads();
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < VT / 32; ++w) t += red[w];
  return t;
}

__device__ __forceinline__ double part_sum(const double* part, int np) {
  double s = 0.0;
  for (int i = threadIdx.x; i < np; i += VT) s += part[i];
  return block_sum(s);
}

// part[c gridDim.x + block] = the block's share of x . y (and of w . y behind all
// of those); COPY: also p = y
template <bool TWO, bool COPY>
__global__ void __launch_bounds__(VT) k_pcg_dot(const double* __restrict__ x,
                                                const double* __restrict__ w,
                                                const double* __restrict__ y, double* p, int64_t N,
                                                double* part) {
  const int64_t off = (int64_t)blockIdx.y * N;
  double s = 0.0, t = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x; i < N; i += (int64_t)gridDim.x * VT) {
    const double v = y[off + i];
    s += x[off + i] * v;
    if (TWO) t += w[off + i] * v;
    if (COPY) p[off + i] = v;
  }
  s = block_sum(s);
  if (TWO) t = block_sum(t);
  if (threadIdx.x == 0) {
    part[blockIdx.y * gridDim.x + blockIdx.x] = s;
    if (TWO) part[(gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(VT) k_pcg_matvec(const double* __restrict__ cpl,
                                                   const double* __restrict__ diag, int n,
                                                   int periodic, const double* __restrict__ p,
                                                   double* q, double* part) {
  const int64_t N = (int64_t)n * n * n, off = (int64_t)blockIdx.y * N;
  double s = 0.0;
  for (int64_t j = (int64_t)blockIdx.x * VT + threadIdx.x; j < N; j += (int64_t)gridDim.x * VT) {
    const double v = stencil_apply(stencil_row(cpl, diag, n, periodic, j), p + off, j);
    q[off + j] = v;
    s += p[off + j] * v;
  }
  s = block_sum(s);
  if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = s;
}

__global__ void __launch_bounds__(VT) k_pcg_update(const double* __restrict__ p,
                                                   const double* __restrict__ q, double* u,
                                                   double* r, int64_t N,
                                                   const double* __restrict__ al, double* part) {
  const int64_t off = (int64_t)blockIdx.y * N;
  const double a = al[blockIdx.y];
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x; i < N; i += (int64_t)gridDim.x * VT) {
    u[off + i] += a * p[off + i];
    const double v = r[off + i] - a * q[off + i];
    r[off + i] = v;
    s += v * v;
  }
  s = block_sum(s);
  if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// the sums of a pass, and what follows from them: START rr and done, RZ rz,
// ALPHA al, RR rr, BETA be and rz (r . z - r_old . z = -al q . z)
enum { SUM_START, SUM_RZ, SUM_ALPHA, SUM_RR, SUM_BETA };
__global__ void __launch_bounds__(VT) k_pcg_sum(int what, int np, PcgScalars s) {
  const int c = blockIdx.x;
  const double v = part_sum(s.part + (int64_t)c * np, np);
  const double w = what == SUM_BETA ? part_sum(s.part + (int64_t)(gridDim.x + c) * np, np) : 0.0;
  if (threadIdx.x) return;
  if (what == SUM_START) {
    s.rr[c] = v;
    s.done[c] = v == 0.0;
  } else if (what == SUM_RZ) {
    s.rz[c] = v;
  } else if (what == SUM_ALPHA) {
    s.al[c] = s.done[c] || v == 0.0 ? 0.0 : s.rz[c] / v;
  } else if (what == SUM_RR) {
    s.rr[c] = v;
  } else {
    s.be[c] = s.done[c] || s.rz[c] == 0.0 ? 0.0 : -s.al[c] * w / s.rz[c];
    if (!s.done[c]) s.rz[c] = v;
  }
}

// p = z + beta p (0 for a finished column, so that later updates leave it alone)
__global__ void __launch_bounds__(VT) k_pcg_p(const double* __restrict__ z, double* p, int64_t N,
                                              PcgScalars s) {
  const int64_t off = (int64_t)blockIdx.y * N;
  const double b = s.be[blockIdx.y];
  const bool done = s.done[blockIdx.y] != 0;
  for (int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x; i < N; i += (int64_t)gridDim.x * VT)
    p[off + i] = done ? 0.0 : z[off + i] + b * p[off + i];
}

inline int grid1(int64_t cnt) { return (int)((cnt + VT - 1) / VT); }

}  // namespace

template <typename T>
void vec_gather(const int32_t* idx, int64_t cnt, const T* y, int64_t ys, T* work, int64_t vs,
                int64_t voff, int nrhs, cudaStream_t st) {
  if (cnt == 0) return;
  ProfScope ps("apply_gather", st, 0.0, (double)cnt * (4.0 + 2.0 * sizeof(T) * nrhs));
  k_gather<T><<<grid1(cnt), VT, 0, st>>>(idx, cnt, y, ys, work, vs, voff, nrhs);
  HIF_CHECK_LAUNCH();
}

template <typename T>
void vec_set(const int32_t* g, const int32_t* pos, int64_t cnt, T* y, int64_t ys,
             const T* work, int64_t vs, int nrhs, cudaStream_t st) {
  if (cnt == 0) return;
  ProfScope ps("apply_scatter", st, 0.0, (double)cnt * (8.0 + 2.0 * sizeof(T) * nrhs));
  k_set<T><<<grid1(cnt), VT, 0, st>>>(g, pos, cnt, y, ys, work, vs, nrhs);
  HIF_CHECK_LAUNCH();
}

template <typename T>
void vec_accumulate(const int32_t* tgt, const int64_t* ptr, const int32_t* src, int64_t ntgt,
                    T* y, int64_t ys, const T* work, int64_t vs, int nrhs, cudaStream_t st) {
  if (ntgt == 0) return;
  ProfScope ps("apply_accumulate", st);
  k_acc<T><<<grid1(ntgt), VT, 0, st>>>(tgt, ptr, src, ntgt, y, ys, work, vs, nrhs);
  HIF_CHECK_LAUNCH();
}

template <typename T>
void vec_convert_in(const double* x, T* y, int64_t cnt, cudaStream_t st) {
  if (cnt == 0) return;
  ProfScope ps("convert", st, 0.0, (double)cnt * (8.0 + sizeof(T)));
  k_cin<T><<<grid1(cnt), VT, 0, st>>>(x, y, cnt);
  HIF_CHECK_LAUNCH();
}

template <typename T>
void vec_convert_out(const T* y, double* x, int64_t cnt, cudaStream_t st) {
  if (cnt == 0) return;
  ProfScope ps("convert", st, 0.0, (double)cnt * (8.0 + sizeof(T)));
  k_cout<T><<<grid1(cnt), VT, 0, st>>>(y, x, cnt);
  HIF_CHECK_LAUNCH();
}

void residual(const double* cpl, const double* diag, int n, int periodic, const double* f,
              const double* u, double* r, int nrhs, cudaStream_t st) {
  const int64_t N = (int64_t)n * n * n;
  ProfScope ps("residual", st, 14.0 * N * nrhs, 8.0 * N * (4.0 + 3.0 * nrhs));
  k_residual<<<grid1(N), VT, 0, st>>>(cpl, diag, n, periodic, f, u, r, nrhs);
  HIF_CHECK_LAUNCH();
}

namespace {
// blocks per column: four points per thread, so that small grids have few sums
int pcg_blocks(int64_t N) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(PCG_BLOCKS, (N + 4 * VT - 1) / (4 * VT)));
}
void pcg_sum(int what, int64_t N, int nrhs, const PcgScalars& s, cudaStream_t st) {
  k_pcg_sum<<<nrhs, VT, 0, st>>>(what, pcg_blocks(N), s);
  HIF_CHECK_LAUNCH();
}
}  // namespace

int64_t pcg_part_elems(int64_t N, int nrhs) { return 2 * (int64_t)pcg_blocks(N) * nrhs; }

void pcg_start(const double* r, int64_t N, int nrhs, const PcgScalars& s, cudaStream_t st) {
  ProfScope ps("dots", st, 2.0 * N * nrhs, 8.0 * N * nrhs);
  k_pcg_dot<false, false><<<dim3(pcg_blocks(N), nrhs), VT, 0, st>>>(r, nullptr, r, nullptr, N, s.part);
  HIF_CHECK_LAUNCH();
  pcg_sum(SUM_START, N, nrhs, s, st);
}

void pcg_first_p(const double* r, const double* z, double* p, int64_t N, int nrhs,
                 const PcgScalars& s, cudaStream_t st) {
  ProfScope ps("dots", st, 2.0 * N * nrhs, 24.0 * N * nrhs);
  k_pcg_dot<false, true><<<dim3(pcg_blocks(N), nrhs), VT, 0, st>>>(r, nullptr, z, p, N, s.part);
  HIF_CHECK_LAUNCH();
  pcg_sum(SUM_RZ, N, nrhs, s, st);
}

void pcg_matvec(const double* cpl, const double* diag, int n, int periodic, const double* p,
                double* q, int nrhs, const PcgScalars& s, cudaStream_t st) {
  const int64_t N = (int64_t)n * n * n;
  ProfScope ps("spmv", st, 15.0 * N * nrhs, 8.0 * N * (4.0 + 2.0 * nrhs));
  k_pcg_matvec<<<dim3(pcg_blocks(N), nrhs), VT, 0, st>>>(cpl, diag, n, periodic, p, q, s.part);
  HIF_CHECK_LAUNCH();
  pcg_sum(SUM_ALPHA, N, nrhs, s, st);
}

void pcg_update(const double* p, const double* q, double* u, double* r, int64_t N, int nrhs,
                const PcgScalars& s, cudaStream_t st) {
  ProfScope ps("axpy", st, 6.0 * N * nrhs, 48.0 * N * nrhs);
  k_pcg_update<<<dim3(pcg_blocks(N), nrhs), VT, 0, st>>>(p, q, u, r, N, s.al, s.part);
  HIF_CHECK_LAUNCH();
  pcg_sum(SUM_RR, N, nrhs, s, st);
}

void pcg_next_p(const double* r, const double* q, const double* z, double* p, int64_t N, int nrhs,
                const PcgScalars& s, cudaStream_t st) {
  {
    ProfScope ps("dots", st, 4.0 * N * nrhs, 24.0 * N * nrhs);
    k_pcg_dot<true, false><<<dim3(pcg_blocks(N), nrhs), VT, 0, st>>>(r, q, z, nullptr, N, s.part);
    HIF_CHECK_LAUNCH();
    pcg_sum(SUM_BETA, N, nrhs, s, st);
  }
  ProfScope ps("axpy", st, 2.0 * N * nrhs, 24.0 * N * nrhs);
  k_pcg_p<<<dim3(pcg_blocks(N), nrhs), VT, 0, st>>>(z, p, N, s);
  HIF_CHECK_LAUNCH();
}

#define HIF_INST(T)                                                                           \
  template void vec_gather<T>(const int32_t*, int64_t, const T*, int64_t, T*, int64_t,       \
                              int64_t, int, cudaStream_t);                                   \
  template void vec_set<T>(const int32_t*, const int32_t*, int64_t, T*, int64_t, const T*,   \
                           int64_t, int, cudaStream_t);                                      \
  template void vec_accumulate<T>(const int32_t*, const int64_t*, const int32_t*, int64_t,   \
                                  T*, int64_t, const T*, int64_t, int, cudaStream_t);        \
  template void vec_convert_in<T>(const double*, T*, int64_t, cudaStream_t);                 \
  template void vec_convert_out<T>(const T*, double*, int64_t, cudaStream_t);
HIF_INST(float)
HIF_INST(double)
#undef HIF_INST

}  // namespace hif
