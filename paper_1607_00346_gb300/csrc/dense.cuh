// Batched dense kernels over uneven fronts (host launch wrappers).
#pragma once

#include <vector>

#include "common.cuh"

namespace hif {

constexpr int NB = 64;      // panel width of the partial Cholesky and of the triangular inverse
constexpr int TILE = 64;    // output tile of the trailing update / batched GEMM

// FP64 retry of FP32 fronts (the LDL^T of §2.2 / §2.3 read as Cholesky, redone
// in double when the FP32 one breaks down): a front whose leading-block
// Cholesky meets a pivot d_j with A_jj / d_j > growth (or d_j not positive)
// is refactored entirely in FP64; growth = 0 turns this off (such a pivot
// then fails the factorization with HIF_ERR_NOT_SPD).  *retried counts them;
// tensor_cores: the retry's products may be slices.
struct RetryOpts {
  double growth;
  int64_t* retried;
  bool tensor_cores;
};

// Partial Cholesky of a batch of fronts (§2.2 and §2.3: A_II = L L^T,
// X = L^{-1} A_IN, A_NN -= X^T X).  Fronts must be sorted by p, largest first.
// On return: trailing blocks of K hold the Schur complements, P holds
// [Linv; X^T] (Linv = L^{-1}, lower triangular) for each front.  With
// tensor_cores the deep products run on gemm_tc (FP64: gemm_f64tc).  With retry
// (FP32 only) the host waits once after the leading blocks are factored to
// read the per-front flags.
template <typename T>
void partial_cholesky(const DFront* d_fronts, const DFront* h_fronts, int nfront, T* Karena,
                      T* Parena, int* d_flags, bool tensor_cores, cudaStream_t st,
                      const RetryOpts* retry = nullptr);

// C = beta C + alpha op(A) op(B) on the tensor cores (tcgen05, 3xTF32; see
// tc.cu): GemmOp semantics as gemm_batched, beta 0 or 1, FP32 data.
// `name` labels the launches in the kernel profile.
void gemm_tc(const GemmOp* d_ops, const GemmOp* h_ops, int nops, const float* Abase,
             const float* Bbase, float* Cbase, int* d_flags, cudaStream_t st,
             const char* name = "gemm_tc");

// The same with an FP64 result of FP64 or FP32 operands: 8-bit slices on the
// BF16 tensor cores, exact sums, one rounding per entry (f64tc.cu).  d_kexp: the
// exponents that KB_DOWN and KB_UP products name.
template <typename S>
void gemm_f64tc(const GemmOp* d_ops, const GemmOp* h_ops, int nops, const S* Abase, const S* Bbase,
                double* Cbase, int* d_flags, cudaStream_t st, const char* name,
                const int* d_kexp = nullptr);
// The exponents of the square roots of the fronts' diagonals, front f's from
// f * stride on (0 where a diagonal entry is not positive and finite).
void diag_exponents(const DFront* d_fronts, int nfront, const double* Karena, int* d_kexp, int stride,
                    cudaStream_t st);

// Autotuning of gemm_tc's tile shape: time the variants on the product
// shapes recorded during a tuning factorization (tune.h).
void tune_gemm_from_records(cudaStream_t st);

// C = beta C + alpha op(A) op(B) for a batch of independent problems, on the
// FMA units.
template <typename T>
void gemm_batched(const GemmOp* d_ops, const GemmOp* h_ops, int nops, const T* Abase,
                  const T* Bbase, T* Cbase, cudaStream_t st, const char* name = "gemm_batched");
// FP64 products that go to gemm_f64tc when tensor cores are allowed.
bool f64tc_worth(const GemmOp* h_ops, int nops);
// gemm_batched, or gemm_f64tc (labelled name_tc) for FP64 products worth it.
template <typename T>
void gemm_fma_or_f64tc(const GemmOp* d_ops, const GemmOp* h_ops, int nops, const T* Abase,
                       const T* Bbase, T* Cbase, int* d_flags, bool tensor_cores, cudaStream_t st,
                       const char* name, const char* name_tc, const int* d_kexp = nullptr) {
  if constexpr (sizeof(T) == 8) {
    if (tensor_cores && f64tc_worth(h_ops, nops)) {
      gemm_f64tc<double>(d_ops, h_ops, nops, Abase, Bbase, Cbase, d_flags, st, name_tc, d_kexp);
      return;
    }
  }
  gemm_batched<T>(d_ops, h_ops, nops, Abase, Bbase, Cbase, st, name);
}

// Mat-vecs of the apply sweeps, y = alpha op(M) x (+ y) batched over GemvOps
// (gemv.cu).  trans = 0: y (rows) = M x; trans = 1: y (cols) = M^T x.
// gemv_plan cuts a list into tasks (a row tile of M x, a column group of
// M^T x); of M x, cnt[k] tiles, in this order, are shared by 8, 4, 2 and 1
// warps; M^T x has one task per thread block (cnt[0]).
struct GemvTask {
  int32_t op, tile;
};
void gemv_plan(const GemvOp* ops, int nops, int trans, std::vector<GemvTask>& tasks, int (&cnt)[4]);
// Thread blocks that run a planned list.
int gemv_ctas(const int (&cnt)[4]);
// Right-hand sides the next block takes when `left` remain, for words of 4
// bytes: 16 (also for 9-15, the others masked), 8 (5-7), 4 (3), 2 or 1, so that
// each block reads the factor once; of 8 bytes, where the multiply-adds of
// masked columns would cost more than a second read: 8, 4, 2 or 1.
int gemv_block(int left, size_t word);

// A planned list and its block of right-hand sides: matrices at M + op.M,
// vectors at w + op.x and w + op.y, nv columns vs apart.
template <typename T>
struct GemvList {
  const GemvOp* ops;
  const GemvTask* tasks;
  const T* M;
  T* w;
  int64_t vs;
  int cnt[4];
  int nv;
};

// A list (ops, tasks, M, w, vs, cnt of `list`) for nrhs right-hand sides.
template <typename T>
void gemv_batched(const GemvOp* h_ops, int nops, const GemvList<T>& list, int trans, int nrhs,
                  cudaStream_t st);

}  // namespace hif
