// Interpolative decomposition from the Gram matrix (pchol.cu).
#pragma once

#include "common.cuh"
#include "front.cuh"

namespace hif {

// Whether fronts of up to nFmax DOFs fit one cluster (one column per thread, 16
// CTAs of 256) and G resolves pivots down to eps.
bool gram_id_fits(int nFmax, double eps);
// Column-pivoted R factor of the fronts' gathered rows (nR x nF blocks of the
// gather arena below the nF x nF ones), stopped at |R_ii| <= eps |R_11|: R (row l of
// column c, leading dimension nF) to Rout + idoff, the permutation and the rank
// as interpolative_decomposition leaves them (T follows in id_solve_t).
// Synchronises the stream once per 64 pivots.
void gram_id(SkelDesc* d_f, const SkelDesc* h_f, int nf, const float* Garena, float* Rout,
             int32_t* perm, double eps, int* d_flags, cudaStream_t st);

}  // namespace hif
