// Vector kernels of the apply sweeps and of the preconditioned solve.
#pragma once

#include "common.cuh"

namespace hif {

// work[q*vs + voff + i] = y[q*ys + idx[i]]
template <typename T>
void vec_gather(const int32_t* idx, int64_t cnt, const T* y, int64_t ys, T* work, int64_t vs,
                int64_t voff, int nrhs, cudaStream_t st);
// y[q*ys + g[i]] = work[q*vs + pos[i]]
template <typename T>
void vec_set(const int32_t* g, const int32_t* pos, int64_t cnt, T* y, int64_t ys,
             const T* work, int64_t vs, int nrhs, cudaStream_t st);
// y[q*ys + tgt[t]] -= sum_{e = ptr[t]}^{ptr[t+1]-1} work[q*vs + src[e]]  (fixed order)
template <typename T>
void vec_accumulate(const int32_t* tgt, const int64_t* ptr, const int32_t* src, int64_t ntgt,
                    T* y, int64_t ys, const T* work, int64_t vs, int nrhs, cudaStream_t st);
// y = (T) x
template <typename T>
void vec_convert_in(const double* x, T* y, int64_t cnt, cudaStream_t st);
// x = (double) y
template <typename T>
void vec_convert_out(const T* y, double* x, int64_t cnt, cudaStream_t st);

// r = f - A u for nrhs columns of length n^3 (seven-point operator, double;
// periodic: neighbours wrap around).
void residual(const double* cpl, const double* diag, int n, int periodic, const double* f,
              const double* u, double* r, int nrhs, cudaStream_t st);

// ---- the vector steps of the conjugate gradients --------------------------------
// Scalars of nrhs columns on the device: the iteration's coefficients are formed
// there, so the host waits once per iteration, for rr.
struct PcgScalars {
  double* rz;    // r . z
  double* al;    // r . z / p . q, 0 for a finished column
  double* be;    // see pcg_next_p, 0 for a finished column
  double* rr;    // r . r
  int* done;     // finished columns (kept by the caller, except the start's)
  double* part;  // pcg_part_elems(N, nrhs) partial sums
};
int64_t pcg_part_elems(int64_t N, int nrhs);
// rr = r . r; done = (rr == 0)
void pcg_start(const double* r, int64_t N, int nrhs, const PcgScalars& s, cudaStream_t st);
// p = z, rz = r . z
void pcg_first_p(const double* r, const double* z, double* p, int64_t N, int nrhs,
                 const PcgScalars& s, cudaStream_t st);
// q = A p, al = rz / p . q
void pcg_matvec(const double* cpl, const double* diag, int n, int periodic, const double* p,
                double* q, int nrhs, const PcgScalars& s, cudaStream_t st);
// u += al p, r -= al q, rr = r . r
void pcg_update(const double* p, const double* q, double* u, double* r, int64_t N, int nrhs,
                const PcgScalars& s, cudaStream_t st);
// beta = (r . z - r_old . z) / rz (Polak-Ribiere) with r_old = r + al q, rz = r . z,
// p = z + beta p (0 for a finished column)
void pcg_next_p(const double* r, const double* q, const double* z, double* p, int64_t N, int nrhs,
                const PcgScalars& s, cudaStream_t st);

}  // namespace hif
