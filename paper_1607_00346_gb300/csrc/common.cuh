// Internal definitions shared by the HIF CUDA translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <utility>

#include "../../include/hif.h"

namespace hif {

// ---- error plumbing ---------------------------------------------------------

struct Error {
  hif_status code;
  std::string msg;
};

void set_last_error(const std::string& msg);

#define HIF_CUDA_TRY(expr)                                                        \
  do {                                                                            \
    cudaError_t e_ = (expr);                                                      \
    if (e_ != cudaSuccess) {                                                      \
      throw ::hif::Error{e_ == cudaErrorMemoryAllocation ? HIF_ERR_OOM            \
                                                          : HIF_ERR_CUDA,         \
                         std::string(#expr) + ": " + cudaGetErrorString(e_)};     \
    }                                                                             \
  } while (0)

// Every kernel launch is followed by HIF_CHECK_LAUNCH(), which also counts it.
int64_t& launch_counter();
// Profiling: while hif_profile_begin() is in force, a ProfScope records CUDA
// events around the launches made during its lifetime, attributed to `name`
// with the given algorithmic flops and bytes.
bool prof_enabled();
// Add algorithmic counts to a kernel's record without a launch (used when the
// counts are only known after the launch, e.g. the ranks found by the ID).
void prof_add(const char* name, double flops, double bytes);
// A scope also counts the kernels launched inside it (this thread's launch
// counter; a CUDA graph replay adds the kernels of the graph).  While a
// ProfSuspend is alive on this thread (a stream capture), scopes record
// nothing.
class ProfScope {
 public:
  ProfScope(const char* name, cudaStream_t st, double flops = 0.0, double bytes = 0.0);
  ~ProfScope();
  ProfScope(const ProfScope&) = delete;
  ProfScope& operator=(const ProfScope&) = delete;

 private:
  cudaStream_t st_;
  bool active_;
  cudaEvent_t a_ = nullptr, b_ = nullptr;
  std::string name_;
  double flops_ = 0.0, bytes_ = 0.0;
  int64_t k0_ = 0;
};
class ProfSuspend {
 public:
  ProfSuspend();
  ~ProfSuspend();
  ProfSuspend(const ProfSuspend&) = delete;
  ProfSuspend& operator=(const ProfSuspend&) = delete;

 private:
  bool prev_;
};

#define HIF_CHECK_LAUNCH()                 \
  do {                                     \
    ++::hif::launch_counter();             \
    HIF_CUDA_TRY(cudaGetLastError());      \
  } while (0)

// ---- device memory --------------------------------------------------------------

// Device bytes of a factor and its factorization: now, and the most so far.
struct MemStats {
  size_t cur = 0, peak = 0;
  void add(size_t bytes) {
    cur += bytes;
    peak = std::max(peak, cur);
  }
};

// Where this thread's factorization counts its kernels' work space (null: nowhere).
inline MemStats*& scratch_stats() {
  static thread_local MemStats* ms = nullptr;
  return ms;
}
class ScratchScope {
 public:
  explicit ScratchScope(MemStats* ms) : prev_(scratch_stats()) { scratch_stats() = ms; }
  ~ScratchScope() { scratch_stats() = prev_; }
  ScratchScope(const ScratchScope&) = delete;
  ScratchScope& operator=(const ScratchScope&) = delete;

 private:
  MemStats* prev_;
};

class DevBuf {
 public:
  DevBuf() = default;
  DevBuf(const DevBuf&) = delete;
  DevBuf& operator=(const DevBuf&) = delete;
  DevBuf(DevBuf&& o) noexcept { swap(o); }
  DevBuf& operator=(DevBuf&& o) noexcept {
    release();
    swap(o);
    return *this;
  }
  ~DevBuf() { release(); }
  void alloc(size_t bytes, MemStats* ms) {
    release();
    ms_ = ms;
    if (bytes == 0) return;
    HIF_CUDA_TRY(cudaMalloc(&p_, bytes));
    bytes_ = bytes;
    if (ms_) ms_->add(bytes);
  }
  // Stream-ordered: allocated and later freed in order on `st` (no device
  // synchronisation); for the temporaries of one factorization.
  void alloc_async(size_t bytes, MemStats* ms, cudaStream_t st) {
    release();
    ms_ = ms;
    if (bytes == 0) return;
    HIF_CUDA_TRY(cudaMallocAsync(&p_, bytes, st));
    st_ = st;
    async_ = true;
    bytes_ = bytes;
    if (ms_) ms_->add(bytes);
  }
  // Work space of a kernel: alloc_async counted in scratch_stats().
  template <typename U>
  U* scratch(size_t count, cudaStream_t st) {
    alloc_async(sizeof(U) * std::max<size_t>(1, count), scratch_stats(), st);
    return as<U>();
  }
  void release() {
    if (p_) {
      if (async_) cudaFreeAsync(p_, st_);
      else cudaFree(p_);
      if (ms_) ms_->cur -= bytes_;
    }
    p_ = nullptr;
    bytes_ = 0;
    async_ = false;
  }
  template <typename U>
  U* as() const { return static_cast<U*>(p_); }
  size_t bytes() const { return bytes_; }

 private:
  void swap(DevBuf& o) {
    std::swap(p_, o.p_);
    std::swap(bytes_, o.bytes_);
    std::swap(ms_, o.ms_);
    std::swap(st_, o.st_);
    std::swap(async_, o.async_);
  }
  void* p_ = nullptr;
  size_t bytes_ = 0;
  MemStats* ms_ = nullptr;
  cudaStream_t st_ = nullptr;
  bool async_ = false;
};

// ---- device-side error flags -------------------------------------------------
// Kernels never trap.  A failed Cholesky pivot (not positive or not finite)
// records the front index in flags[FLAG_NOT_SPD] (first failure wins) and the
// kernel carries on with a harmless value so that the launch finishes
// normally; a bounded wait that ran out records the front in
// flags[FLAG_TIMEOUT] and the kernel returns early.
enum : int { FLAG_NOT_SPD = 0, FLAG_TIMEOUT = 1, FLAG_COUNT = 4 };

// ---- work descriptors ---------------------------------------------------------

// A dense front: an n x n column-major frontal matrix K (ld = n) whose first p
// columns are eliminated (partial Cholesky), and an n x p factor panel P
// (ld = n) that receives [Linv; X^T] (Linv = L^{-1} of the leading p x p block).
struct DFront {
  int64_t K;     // element offset of K in the K arena
  int64_t P;     // element offset of P in the factor arena
  int n;         // extent handled by the kernel (rows/columns 0..n-1)
  int p;
  int id;        // front number (reported on failure)
  int ld;        // leading dimension of K and P (the front's full size)
};

// Batched matrix product C (m x n) = beta C + alpha op(A) op(B) with k inner.
// kzero: a triangular operand, whose zeros the kernels leave out tile by tile
// (half of the product): KZ_B_UP op(B)[k][c] = 0 for k > c, KZ_B_LOW
// op(B)[k][c] = 0 for k < c, KZ_A_LOW op(A)[r][k] = 0 for k > r.
enum : int { KZ_NONE = 0, KZ_B_UP = 1, KZ_B_LOW = 2, KZ_A_LOW = 3 };
// kbal: how gemm_f64tc balances the scales of k between the operands (f64tc.cu).
// KB_MAX by their largest entries, KB_NONE not at all, KB_DOWN column k of op(A) times
// 2^-e[ks + k] and row k of op(B) times 2^e[ks + k], KB_UP the other way round.
enum : int { KB_MAX = 0, KB_NONE = 1, KB_DOWN = 2, KB_UP = 3 };
struct GemmOp {
  int64_t A, B, C;   // element offsets from the A, B and C base pointers of the launch
  int m, n, k;
  int lda, ldb, ldc;
  int transA, transB;
  float alpha, beta;
  int lower;         // 1: C is symmetric, only tiles touching its lower triangle are computed
  int kzero;
  int kbal;
  int64_t ks;
};

// The tile a block computes (longest sums first: with a triangular operand the
// tiles of the last columns or rows have them) and the k it has to visit.
__host__ __device__ inline int gemm_tile(const GemmOp& o, int block, int tiles) {
  return o.kzero == KZ_B_UP || o.kzero == KZ_A_LOW ? tiles - 1 - block : block;
}
__host__ __device__ inline void gemm_k_range(const GemmOp& o, int rb, int tr, int cb, int tc,
                                             int* kbeg, int* kend) {
  *kbeg = o.kzero == KZ_B_LOW ? cb : 0;
  const int e = o.kzero == KZ_B_UP ? cb + tc : o.kzero == KZ_A_LOW ? rb + tr : o.k;
  *kend = e < o.k ? e : o.k;
  if (*kbeg > *kend) *kbeg = *kend;
}

// Batched matrix-vector product on a front of the apply (see apply kernels).
struct GemvOp {
  int64_t M;      // element offset of the matrix in the factor arena
  int64_t x;      // offset of the input vector in the work arena
  int64_t y;      // offset of the output vector in the work arena
  int rows, cols; // matrix shape (column-major)
  int ld;
  int tri;        // 1: matrix is lower triangular (only r >= c read)
  float alpha;
  int beta_one;   // 1: y += alpha op(M) x ; 0: y = alpha op(M) x
};

inline int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

}  // namespace hif
