// Batched dense kernels over uneven fronts: partial Cholesky (panel factor +
// triangular solve + trailing rank-NB update), inverse of the Cholesky factor
// and the generic batched GEMM.
//
// Every kernel takes a descriptor array (one entry per front or problem) and a
// 2-D grid: blockIdx.y = descriptor, blockIdx.x = tile / chunk inside it.
// Fronts whose work is finished, and tiles outside a front, exit at once.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <type_traits>
#include <vector>

#include "dense.cuh"

namespace hif {

namespace {

constexpr int KC = 16;            // inner-dimension chunk of the tile products
constexpr int MAX_GRID_Y = 65535;

__device__ __forceinline__ void flag_front(int* flags, int which, int id) {
  atomicCAS(&flags[which], -1, id);
}

// ---- tile micro-kernel ---------------------------------------------------------
// 256 threads, 64 x 64 output, thread t owns rows (t % 16)*4 .. +4 and columns
// (t / 16)*4 .. +4.  As[k][r] and Bs[k][c] hold a KC-deep slice.
template <typename T>
struct TileAcc {
  T v[4][4];
  __device__ void zero() {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[i][j] = T(0);
  }
  __device__ void mma(const T (*As)[TILE + 4], const T (*Bs)[TILE + 4], int kdepth) {
    const int tr = (threadIdx.x % 16) * 4, tc = (threadIdx.x / 16) * 4;
    for (int k = 0; k < kdepth; ++k) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[k][tr + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[k][tc + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) v[i][j] = fma(a[i], b[j], v[i][j]);
    }
  }
};

// ---- one step of the leading-block Cholesky: diagonal block, panel, update -----
// What bounds a step is its chain: the fronts of the upper levels are few, so
// the three kernels run one after the other with most of the chip idle.
//
// k_chol_diag: one CTA per front factors the jb x jb diagonal block (jb <= 64) in
// shared memory, 16 columns at a time: one warp factors the 16 x 16 block in
// registers (rows across lanes, pivot column by shuffles), four threads per row solve
// the rows below and, in the same pass, the block's own inverse, all threads update
// the rest; three CTA barriers per 16 columns.  The inverses are merged pairwise to 32
// and 64 and L^{-1} left in the factor panel, zeros above the diagonal: the panel below
// becomes a product, and the triangular inverse of the whole front needs these blocks
// anyway.  In FP64 an instruction of one warp takes 64 clocks (each quarter of an SM
// has a quarter of its FP64 unit), masked or not: so every phase but the factoring
// warp's spreads over all quarters, without masked multiply-adds.  Clocks of a 64-column
// block in FP64, before and after that: factor 69 k -> 63 k, solve and 16-wide inverses
// 43 k -> 25 k, update 39 k -> 23 k, merges 50 k -> 41 k.
// 64 columns, FP32 25 us, FP64 100 -> 77 us: with one column per barrier pair and no
// inverse 62 and 112 us; the panel below 8 us (by substitution 30-37, FP64 117), the
// 64-deep update of one tile 11 us (18, FP64 49), and the separate inverse took 25-95 us.
//
// A non-positive or non-finite pivot flags the front and continues with 1.  With
// growth > 0 (FP32 fronts that may be retried in FP64), the panel's diagonal
// holds the front's original diagonal A_jj on entry, and a pivot d_j with
// A_jj / d_j > growth (cancellation has eaten all but a few bits of it), or one
// that is not positive or not finite, marks the front in fflag[blockIdx.x]
// instead of failing it.
constexpr int CB = 16;             // columns factored per step of the diagonal block
constexpr int DP = NB + 1;         // row pitch of the shared-memory blocks

template <typename T>
constexpr size_t chol_diag_smem() {
  return sizeof(T) * 2 * NB * DP;
}

// 1 / sqrt(d) (in FP32 with one Newton step): every column of the block waits for it.
__device__ __forceinline__ float inverse_root(float d) {
  const float y = rsqrtf(d);
  return fmaf(0.5f * y, fmaf(-d * y, y, 1.0f), y);
}
__device__ __forceinline__ double inverse_root(double d) { return rsqrt(d); }
// d positive and finite (the double without the FP64 unit)
__device__ __forceinline__ bool pivot_ok(float d) { return d > 0.f && isfinite(d); }
__device__ __forceinline__ bool pivot_ok(double d) {
  const long long b = __double_as_longlong(d);
  return b > 0 && b < 0x7ff0000000000000ll;
}

// S(i, j) -= X_i X_j^T over the N blocks of 16 rows below the block at o.  The number
// of blocks is a template argument: masked multiply-adds take their turn on the FP64
// unit like the others.
template <int N, typename T>
__device__ __forceinline__ void chol_diag_update(T (*S)[DP], int o) {
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  T u[N * (N + 1) / 2];
#pragma unroll
  for (int i = 0; i < N * (N + 1) / 2; ++i) u[i] = T(0);
#pragma unroll
  for (int l = 0; l < CB; ++l) {
    T xr[N], xc[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      xr[i] = S[o + CB + ty + 16 * i][o + l];
      xc[i] = S[o + CB + tx + 16 * i][o + l];
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int j = 0; j <= i; ++j)
        u[i * (i + 1) / 2 + j] = fma(xr[i], xc[j], u[i * (i + 1) / 2 + j]);
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j <= i; ++j)
      S[o + CB + ty + 16 * i][o + CB + tx + 16 * j] -= u[i * (i + 1) / 2 + j];
}

template <typename T>
__global__ void __launch_bounds__(256) k_chol_diag(const DFront* __restrict__ fr, const T* Kar,
                                                   T* Par, int j0, int* flags, float growth,
                                                   int* fflag) {
  const DFront d = fr[blockIdx.x];
  if (j0 >= d.p) return;
  const int jb = min(NB, d.p - j0);
  const int64_t ld = d.ld;
  const T* K = Kar + d.K + (int64_t)j0 + (int64_t)j0 * ld;
  T* P = Par + d.P + (int64_t)j0 + (int64_t)j0 * ld;
  extern __shared__ __align__(16) unsigned char dsm[];
  T(*S)[DP] = reinterpret_cast<T(*)[DP]>(dsm);                       // A, then L
  T(*V)[DP] = reinterpret_cast<T(*)[DP]>(dsm + sizeof(T) * NB * DP);  // L^{-1}
  __shared__ T s_inv[NB], s_orig[NB];
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int nb16 = (jb + CB - 1) / CB, je = nb16 * CB;
  // lower triangle, padded to whole 16-blocks with the identity
  for (int e = tid; e < NB * je; e += 256) {
    const int r = e % NB, c = e / NB;
    if (r < je) S[r][c] = (r < jb && c < jb && r >= c) ? K[r + (int64_t)c * ld] : T(r == c ? 1 : 0);
  }
  if (growth > 0.f && tid < jb) s_orig[tid] = P[tid + (int64_t)tid * ld];
  __syncthreads();
  for (int o = 0; o < je; o += CB) {
    if (warp == 0) {
      // lane (r, h): the entries of row r in columns 2 u + h
      const int r = lane % CB, h = lane / CB;
      T a[CB / 2];
#pragma unroll
      for (int u = 0; u < CB / 2; ++u) a[u] = 2 * u + h <= r ? S[o + r][o + 2 * u + h] : T(0);
      bool bad = false, weak = false;
      T myinv = T(0);
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        T dv = __shfl_sync(0xffffffffu, a[c / 2], c + (c % 2) * CB);
        const bool ok = pivot_ok(dv);
        if (o + c < jb) {
          bad = bad || !ok;
          if (growth > 0.f) weak = weak || !ok || dv * (T)growth < s_orig[o + c];
        }
        if (!ok) dv = T(1);
        const T inv = inverse_root(dv);
        // column c of L, in every lane of row r
        const T ac = __shfl_sync(0xffffffffu, a[c / 2], r + (c % 2) * CB);
        T l;   // in FP64 one product fewer (64 clocks), in FP32 a shorter chain
        if constexpr (sizeof(T) == 8) l = r >= c ? (r == c ? dv : ac) * inv : T(0);
        else l = r > c ? ac * inv : (r == c ? dv * inv : T(0));
        if (h == c % 2) a[c / 2] = l;
        if (r == c) myinv = inv;
#pragma unroll
        for (int u = (c + 1) / 2; u < CB / 2; ++u) {
          const T lj = __shfl_sync(0xffffffffu, l, 2 * u + h);
          if (2 * u + h > c) a[u] = fma(-l, lj, a[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < CB / 2; ++u) S[o + r][o + 2 * u + h] = 2 * u + h <= r ? a[u] : T(0);
      if (h == 0) s_inv[o + r] = myinv;
      if (lane == 0) {
        if (growth > 0.f) {
          if (weak) fflag[blockIdx.x] = 1;
        } else if (bad) {
          flag_front(flags, FLAG_NOT_SPD, d.id);
        }
      }
    }
    __syncthreads();
    // rows below: X L_oo^T = A; and 16 rows of the identity, which become L_oo^{-T}:
    // four threads per row (thread t: columns t + 4 q), so that all four parts of the
    // SM have a share
    const int below = je - o - CB;
    if (tid / 4 < below + CB) {   // whole warps
      const int rr = tid / 4, t = tid % 4, e = rr - below;
      T x[CB / 4];
#pragma unroll
      for (int q = 0; q < CB / 4; ++q)
        x[q] = e >= 0 ? T(t + 4 * q == e ? 1 : 0) : S[o + CB + rr][o + t + 4 * q];
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const T xc = __shfl_sync(0xffffffffu, x[c / 4] * s_inv[o + c], (lane & 28) | (c % 4));
        if (t == c % 4) x[c / 4] = xc;
#pragma unroll
        for (int q = c / 4 + (c % 4 == 3); q < CB / 4; ++q)
          if (t + 4 * q > c) x[q] = fma(-xc, S[o + t + 4 * q][o + c], x[q]);
      }
#pragma unroll
      for (int q = 0; q < CB / 4; ++q) {
        if (e >= 0) V[o + t + 4 * q][o + e] = x[q];
        else S[o + CB + rr][o + t + 4 * q] = x[q];
      }
    }
    __syncthreads();
    if (below == 0) break;
    // rank-16 update of the lower triangle of the rest: thread (ty, tx) of a
    // 16 x 16 grid takes one entry of each 16 x 16 block
    if (below == 3 * CB) chol_diag_update<3>(S, o);
    else if (below == 2 * CB) chol_diag_update<2>(S, o);
    else chol_diag_update<1>(S, o);
    __syncthreads();
  }
  // pairs of blocks of w: [A 0; B C]^-1 = [A^-1 0; -C^-1 B A^-1  C^-1].  B A^-1 is
  // kept transposed in the free block above the diagonal.
  for (int w = CB; w < je; w *= 2) {
    // 2 x 2 entries per thread: w = 16 has up to two pairs (128 threads), w = 32
    // one (256); rows past je (a shorter right block) are computed and unused
    const int per = w * w / 4, q = tid / per, o = 2 * w * q;
    // the depth goes with 2 g, down or up: equal g in a half warp, and the two warps
    // of one part of the SM (warp and warp + 4) from opposite ends
    const int l = tid % per % (w / 2);
    const int g = w == 32 ? (warp < 4 ? warp : 11 - warp) * 2 + lane / 16 : tid % per / (w / 2);
    int r = 2 * l, c = 2 * g;
    if (o + w + r < je) {
      T t00 = T(0), t01 = T(0), t10 = T(0), t11 = T(0);
#pragma unroll 8
      for (int k = c; k < w; ++k) {   // V[o + k][o + c] is zero for k < c
        const T s0 = S[o + w + r][o + k], s1 = S[o + w + r + 1][o + k];
        const T v0 = V[o + k][o + c], v1 = V[o + k][o + c + 1];
        t00 = fma(s0, v0, t00);
        t01 = fma(s0, v1, t01);
        t10 = fma(s1, v0, t10);
        t11 = fma(s1, v1, t11);
      }
      V[o + c][o + w + r] = t00;
      V[o + c + 1][o + w + r] = t01;
      V[o + c][o + w + r + 1] = t10;
      V[o + c + 1][o + w + r + 1] = t11;
    }
    __syncthreads();
    r = 2 * g;
    c = 2 * l;
    if (o + w + r < je) {
      T t00 = T(0), t01 = T(0), t10 = T(0), t11 = T(0);
#pragma unroll 8
      for (int k = 0; k <= r + 1; ++k) {
        const T v0 = V[o + w + r][o + w + k], v1 = V[o + w + r + 1][o + w + k];
        const T s0 = V[o + c][o + w + k], s1 = V[o + c + 1][o + w + k];
        t00 = fma(v0, s0, t00);
        t01 = fma(v0, s1, t01);
        t10 = fma(v1, s0, t10);
        t11 = fma(v1, s1, t11);
      }
      V[o + w + r][o + c] = -t00;
      V[o + w + r][o + c + 1] = -t01;
      V[o + w + r + 1][o + c] = -t10;
      V[o + w + r + 1][o + c + 1] = -t11;
    }
    __syncthreads();
  }
  for (int e = tid; e < NB * jb; e += 256) {
    const int r = e % NB, c = e / NB;
    if (r < jb) P[r + (int64_t)c * ld] = r >= c ? V[r][c] : T(0);
  }
}

// 64 x 64 tiles with the whole depth of 64 in shared memory: one load phase, one
// barrier, 64 steps.  Xs[k][i], Ys[k][j]; thread t owns rows (t % 16) 4 .. and
// columns (t / 16) 4 ..
constexpr int SP = TILE + 4;       // row pitch: 16-byte rows
template <typename T>
constexpr size_t step_smem() {
  return sizeof(T) * 2 * NB * SP;
}
template <typename T>
__device__ __forceinline__ void step_mma(const T (*Xs)[SP], const T (*Ys)[SP], int depth,
                                         T (&v)[4][4]) {
  const int tr = (threadIdx.x % 16) * 4, tc = (threadIdx.x / 16) * 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = T(0);
#pragma unroll 4
  for (int k = 0; k < depth; ++k) {
    T x[4], y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[i] = Xs[k][tr + i];
      y[i] = Ys[k][tc + i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[i][j] = fma(x[i], y[j], v[i][j]);
  }
}

// k_panel: the rows below the diagonal block, L21 = A21 L11^{-T}, in place (a CTA
// owns 64 rows of all 64 columns; only fronts with a full block have rows below).
// L11^{-1} is lower triangular: column c sums k <= c.
template <typename T>
__global__ void __launch_bounds__(256) k_panel(const DFront* __restrict__ fr, T* Kar,
                                               const T* __restrict__ Par, int j0) {
  const DFront d = fr[blockIdx.y];
  const int j1 = j0 + NB;
  const int r0 = j1 + blockIdx.x * TILE;
  if (r0 >= d.n) return;
  const int64_t ld = d.ld;
  T* K = Kar + d.K + (int64_t)j0 * ld;
  const T* P = Par + d.P + (int64_t)j0 + (int64_t)j0 * ld;
  extern __shared__ __align__(16) unsigned char ssm[];
  T(*Xs)[SP] = reinterpret_cast<T(*)[SP]>(ssm);
  T(*Ys)[SP] = Xs + NB;
#pragma unroll 8
  for (int e = threadIdx.x; e < NB * TILE; e += 256) {
    const int r = e % TILE, k = e / TILE;
    Xs[k][r] = r0 + r < d.n ? K[r0 + r + (int64_t)k * ld] : T(0);
    Ys[k][r] = P[r + (int64_t)k * ld];
  }
  __syncthreads();
  T v[4][4];
  step_mma<T>(Xs, Ys, (threadIdx.x / 16) * 4 + 4, v);
  const int tr = (threadIdx.x % 16) * 4, tc = (threadIdx.x / 16) * 4;
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (r0 + tr + i < d.n) K[r0 + tr + i + (int64_t)(tc + j) * ld] = v[i][j];
}

__device__ __forceinline__ void tri_index(int t, int& ti, int& tj) {
  int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (i * (i + 1) / 2 > t) --i;
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  ti = i;
  tj = t - i * (i + 1) / 2;
}

// ---- trailing update: K[j1:n, j1:n] -= K[j1:n, j0:j1] K[j1:n, j0:j1]^T (lower tiles)
// (jmax < n: only the columns below jmax, i.e. the rest of an outer block;
// the tiles then form nrow x ncol rectangles, strictly upper ones skipped)
template <typename T>
__global__ void __launch_bounds__(256) k_syrk(const DFront* __restrict__ fr, T* Kar, int j0,
                                              int jmax) {
  const DFront d = fr[blockIdx.y];
  const int j1 = j0 + NB;   // a front with rows below has a full block
  const int n = d.n;
  if (j1 >= n) return;
  const int64_t ld = d.ld;
  const int nt = (n - j1 + TILE - 1) / TILE;
  int ti, tj;
  if (jmax >= n) {
    if ((int)blockIdx.x >= nt * (nt + 1) / 2) return;
    tri_index(blockIdx.x, ti, tj);
  } else {
    const int nct = (jmax - j1 + TILE - 1) / TILE;
    if (nct <= 0 || (int)blockIdx.x >= nt * nct) return;
    ti = blockIdx.x % nt;
    tj = blockIdx.x / nt;
    if (tj > ti) return;
  }
  const int rb = j1 + ti * TILE, cb = j1 + tj * TILE;
  T* K = Kar + d.K;
  extern __shared__ __align__(16) unsigned char ssm[];
  T(*Xs)[SP] = reinterpret_cast<T(*)[SP]>(ssm);
  T(*Ys)[SP] = Xs + NB;
#pragma unroll 8
  for (int e = threadIdx.x; e < NB * TILE; e += 256) {
    const int r = e % TILE, k = e / TILE;
    const int64_t o = (int64_t)(j0 + k) * ld;
    Xs[k][r] = rb + r < n ? K[rb + r + o] : T(0);
    Ys[k][r] = cb + r < n ? K[cb + r + o] : T(0);
  }
  // this thread's entries of the tile, loaded before the barrier
  const int tr = (threadIdx.x % 16) * 4, tc = (threadIdx.x / 16) * 4;
  T u[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = rb + tr + i, c = cb + tc + j;
      u[i][j] = r < n && r >= c && c < jmax ? K[(int64_t)r + (int64_t)c * ld] : T(0);
    }
  __syncthreads();
  T v[4][4];
  step_mma<T>(Xs, Ys, NB, v);
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = rb + tr + i, c = cb + tc + j;
      if (r < n && r >= c && c < jmax) K[(int64_t)r + (int64_t)c * ld] = u[i][j] - v[i][j];
    }
}

// ---- FP64 retry of FP32 fronts flagged by the leading-block Cholesky ----------
// Before the leading block is factored: its p x p entries are copied to a
// snapshot S (column-major, ld = p) and its diagonal to the panel's diagonal
// (where k_chol_diag reads the original A_jj).
template <typename T>
__global__ void __launch_bounds__(256) k_retry_prep(const DFront* __restrict__ fr, const T* Kar,
                                                    T* Par, T* S, const int64_t* __restrict__ soff) {
  const DFront d = fr[blockIdx.y];
  const int64_t pp = (int64_t)d.p * d.p;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < pp; e += (int64_t)gridDim.x * 256) {
    const int r = (int)(e % d.p), c = (int)(e / d.p);
    const T v = Kar[d.K + r + (int64_t)c * d.ld];
    S[soff[blockIdx.y] + e] = v;
    if (r == c) Par[d.P + r + (int64_t)c * d.ld] = v;
  }
}

// A flagged front in the FP32 arenas and its FP64 copy.
struct RetryMap {
  int64_t Kf, Pf;   // offsets in the FP32 K and panel arenas
  int64_t Kd, Pd;   // offsets in the FP64 copies
  int64_t S;        // offset of its leading-block snapshot
  int p, ld;        // eliminated count, size (= leading dimension)
};

// FP64 copy of the original front: the leading block from the snapshot, the
// rest (A_NI, A_NN: untouched by the leading-block Cholesky) from K.
__global__ void __launch_bounds__(256) k_retry_build(const RetryMap* __restrict__ mp,
                                                     const float* Kar, const float* S,
                                                     double* Kd) {
  const RetryMap m = mp[blockIdx.y];
  const int64_t tot = (int64_t)m.ld * m.ld;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < tot; e += (int64_t)gridDim.x * 256) {
    const int r = (int)(e % m.ld), c = (int)(e / m.ld);
    const float v = (r < m.p && c < m.p) ? S[m.S + r + (int64_t)c * m.p] : Kar[m.Kf + e];
    Kd[m.Kd + e] = (double)v;
  }
}

// Results of the FP64 partial Cholesky back in FP32: the whole panel
// [Linv; X^T] and the Schur complement (trailing block of K).
__global__ void __launch_bounds__(256) k_retry_writeback(const RetryMap* __restrict__ mp,
                                                         const double* Kd, const double* Pd,
                                                         float* Kar, float* Par) {
  const RetryMap m = mp[blockIdx.y];
  const int64_t np = (int64_t)m.ld * m.p;
  const int nb = m.ld - m.p;
  const int64_t nn = (int64_t)nb * nb;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < np + nn;
       e += (int64_t)gridDim.x * 256) {
    if (e < np) {
      Par[m.Pf + e] = (float)Pd[m.Pd + e];
    } else {
      const int64_t q = e - np;
      const int r = m.p + (int)(q % nb), c = m.p + (int)(q / nb);
      const int64_t o = r + (int64_t)c * m.ld;
      Kar[m.Kf + o] = (float)Kd[m.Kd + o];
    }
  }
}

__global__ void __launch_bounds__(128) k_diag_exponents(const DFront* __restrict__ fr,
                                                       const double* __restrict__ Kar, int* e,
                                                       int stride) {
  const DFront d = fr[blockIdx.x];
  for (int i = threadIdx.x; i < d.n; i += 128) {
    const double v = Kar[d.K + i + (int64_t)i * d.ld];
    e[(int64_t)blockIdx.x * stride + i] = v > 0.0 && isfinite(v) ? ilogb(v) >> 1 : 0;
  }
}

// ---- generic batched GEMM ------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_gemm(const GemmOp* __restrict__ ops, const T* Ab,
                                              const T* Bb, T* Cb) {
  const GemmOp o = ops[blockIdx.y];
  const int tm = (o.m + TILE - 1) / TILE, tn = (o.n + TILE - 1) / TILE;
  if ((int)blockIdx.x >= tm * tn) return;
  const int tile = gemm_tile(o, blockIdx.x, tm * tn);
  const int rb = (tile % tm) * TILE, cb = (tile / tm) * TILE;
  if (o.lower && cb >= rb + TILE) return;
  int kbeg, kend;
  gemm_k_range(o, rb, TILE, cb, TILE, &kbeg, &kend);
  const T* A = Ab + o.A;
  const T* B = Bb + o.B;
  T* C = Cb + o.C;
  __shared__ T As[KC][TILE + 4];
  __shared__ T Bs[KC][TILE + 4];
  TileAcc<T> acc;
  acc.zero();
  for (int k0 = kbeg; k0 < kend; k0 += KC) {
    for (int e = threadIdx.x; e < KC * TILE; e += 256) {
      int rr, kk;
      // choose the thread mapping that reads memory contiguously
      if (!o.transA) { rr = e % TILE; kk = e / TILE; } else { kk = e % KC; rr = e / KC; }
      int r = rb + rr, k = k0 + kk;
      T v = T(0);
      if (r < o.m && k < o.k)
        v = o.transA ? A[(int64_t)k + (int64_t)r * o.lda] : A[(int64_t)r + (int64_t)k * o.lda];
      As[kk][rr] = v;
      int cc;
      if (o.transB) { cc = e % TILE; kk = e / TILE; } else { kk = e % KC; cc = e / KC; }
      int c = cb + cc;
      k = k0 + kk;
      v = T(0);
      if (c < o.n && k < o.k)
        v = o.transB ? B[(int64_t)c + (int64_t)k * o.ldb] : B[(int64_t)k + (int64_t)c * o.ldb];
      Bs[kk][cc] = v;
    }
    __syncthreads();
    acc.mma(As, Bs, KC);
    __syncthreads();
  }
  const int tr = (threadIdx.x % 16) * 4, tc = (threadIdx.x / 16) * 4;
  const T alpha = (T)o.alpha, beta = (T)o.beta;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = cb + tc + j;
    if (c >= o.n) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = rb + tr + i;
      if (r >= o.m) continue;
      T* cp = &C[(int64_t)r + (int64_t)c * o.ldc];
      *cp = (beta == T(0) ? T(0) : beta * *cp) + alpha * acc.v[i][j];
    }
  }
}

}  // namespace

// ---- host wrappers ---------------------------------------------------------------

// products at least this large (rows of X^T) go to the tensor cores (FP32)
constexpr int TC_MIN_ROWS = 256;

template <typename T>
void finish_fronts(const DFront* d_fronts, const DFront* h_fronts, int nfront, T* Karena,
                   T* Parena, int* d_flags, bool tensor_cores, cudaStream_t st, const int* d_kexp,
                   int kstride);

// Refactor the flagged FP32 fronts entirely in FP64 (from the snapshot of
// their leading blocks and their untouched A_NI, A_NN) and store the results
// in the FP32 arenas.
static void retry_fronts_fp64(const std::vector<int>& bad, const DFront* h_fronts,
                       const std::vector<int64_t>& soff, float* Karena, float* Parena,
                       const float* snap, int* d_flags, bool tensor_cores, cudaStream_t st) {
  const int nb = (int)bad.size();
  std::vector<DFront> dl;
  std::vector<RetryMap> maps;
  int64_t kt = 0, pt = 0, mx = 0;
  for (int f : bad) {
    const DFront& h = h_fronts[f];
    dl.push_back(DFront{kt, pt, h.n, h.p, h.id, h.ld});
    maps.push_back(RetryMap{h.K, h.P, kt, pt, soff[f], h.p, h.ld});
    kt += (int64_t)h.ld * h.ld;
    pt += (int64_t)h.ld * h.p;
    mx = std::max<int64_t>(mx, (int64_t)h.ld * h.ld);
  }
  DevBuf Kb, Pb, maps_b, dl_b;
  double* Kd = Kb.scratch<double>(kt, st);
  double* Pd = Pb.scratch<double>(pt, st);
  RetryMap* d_maps = maps_b.scratch<RetryMap>(nb, st);
  DFront* d_dl = dl_b.scratch<DFront>(nb, st);
  HIF_CUDA_TRY(cudaMemsetAsync(Pd, 0, sizeof(double) * std::max<int64_t>(1, pt), st));
  HIF_CUDA_TRY(cudaMemcpyAsync(d_maps, maps.data(), sizeof(RetryMap) * nb, cudaMemcpyHostToDevice, st));
  HIF_CUDA_TRY(cudaMemcpyAsync(d_dl, dl.data(), sizeof(DFront) * nb, cudaMemcpyHostToDevice, st));
  const int gx = std::max(1, std::min(1024, ceil_div(mx, 256)));
  for (int f0 = 0; f0 < nb; f0 += MAX_GRID_Y) {
    const int c = std::min(MAX_GRID_Y, nb - f0);
    ProfScope ps("chol_retry_fp64", st);
    k_retry_build<<<dim3(gx, c), 256, 0, st>>>(d_maps + f0, Karena, snap, Kd);
    HIF_CHECK_LAUNCH();
  }
  partial_cholesky<double>(d_dl, dl.data(), nb, Kd, Pd, d_flags, tensor_cores, st, nullptr);
  for (int f0 = 0; f0 < nb; f0 += MAX_GRID_Y) {
    const int c = std::min(MAX_GRID_Y, nb - f0);
    ProfScope ps("chol_retry_fp64", st);
    k_retry_writeback<<<dim3(gx, c), 256, 0, st>>>(d_maps + f0, Kd, Pd, Karena, Parena);
    HIF_CHECK_LAUNCH();
  }
}

template <typename T>
void partial_cholesky(const DFront* d_fronts, const DFront* h_fronts, int nfront, T* Karena,
                      T* Parena, int* d_flags, bool tensor_cores, cudaStream_t st,
                      const RetryOpts* retry) {
  if (nfront == 0) return;
  const int pmax = h_fronts[0].p;
  // FP32 fronts that may be retried in FP64: snapshot of every leading block,
  // original diagonal in the panel, one flag per front
  const bool growth_on = std::is_same<T, float>::value && retry && retry->growth > 0.0;
  int* d_fflag = nullptr;
  DevBuf snap_b;
  T* snap = nullptr;
  int64_t* d_soff = nullptr;
  std::vector<int64_t> soff;
  if (growth_on) {
    soff.resize(nfront);
    int64_t tot = 0, mx = 1;
    for (int f = 0; f < nfront; ++f) {
      soff[f] = tot;
      tot += (int64_t)h_fronts[f].p * h_fronts[f].p;
      mx = std::max<int64_t>(mx, (int64_t)h_fronts[f].p * h_fronts[f].p);
    }
    HIF_CUDA_TRY(cudaMallocAsync(&d_fflag, sizeof(int) * nfront, st));
    snap = snap_b.scratch<T>(tot, st);
    HIF_CUDA_TRY(cudaMallocAsync(&d_soff, sizeof(int64_t) * nfront, st));
    HIF_CUDA_TRY(cudaMemsetAsync(d_fflag, 0, sizeof(int) * nfront, st));
    HIF_CUDA_TRY(cudaMemcpyAsync(d_soff, soff.data(), sizeof(int64_t) * nfront,
                                 cudaMemcpyHostToDevice, st));
    const int gx = std::max(1, std::min(1024, ceil_div(mx, 256)));
    for (int f0 = 0; f0 < nfront; f0 += MAX_GRID_Y) {
      const int c = std::min(MAX_GRID_Y, nfront - f0);
      ProfScope ps("chol_retry_snapshot", st, 0.0, 2.0 * sizeof(T) * tot);
      k_retry_prep<T><<<dim3(gx, c), 256, 0, st>>>(d_fronts + f0, Karena, Parena, snap, d_soff + f0);
      HIF_CHECK_LAUNCH();
    }
  }
  // 1. Cholesky of the leading p x p block (right-looking, panels of NB):
  //    the kernels see extent p, leading dimension n
  std::vector<DFront> lead(h_fronts, h_fronts + nfront);
  for (auto& f : lead) f.n = f.p;
  DFront* d_lead = nullptr;
  HIF_CUDA_TRY(cudaMallocAsync(&d_lead, sizeof(DFront) * nfront, st));
  HIF_CUDA_TRY(cudaMemcpyAsync(d_lead, lead.data(), sizeof(DFront) * nfront,
                               cudaMemcpyHostToDevice, st));
  // two levels: inner panels of NB factor an outer block of NB2 columns and
  // update only its remaining columns; the rows and columns right of the
  // outer block then get one rank-NB2 update A22 -= L21 L21^T as a batched
  // product (tensor cores for FP32).  FP64 on the tensor cores: a product
  // costs its launches (about 40 us) up to several waves of tiles, so
  // panel and update are one product each over all that is left.
  constexpr int NB2 = 256;
  const bool f64tc = sizeof(T) == 8 && tensor_cores;
  const bool outer = pmax > NB2 && !f64tc;
  DevBuf kexp_b;
  int* d_kexp = nullptr;   // scales of the eliminated DOFs, for the products' k
  const int kstride = f64tc ? pmax : 0;
  if constexpr (sizeof(T) == 8) {
    if (f64tc) {
      d_kexp = kexp_b.scratch<int>((size_t)nfront * kstride, st);
      diag_exponents(d_lead, nfront, Karena, d_kexp, kstride, st);
    }
  }
  static const bool attr = [] {   // initialised once, also under concurrent factorizations
    HIF_CUDA_TRY(cudaFuncSetAttribute(k_chol_diag<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)chol_diag_smem<T>()));
    HIF_CUDA_TRY(cudaFuncSetAttribute(k_panel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)step_smem<T>()));
    HIF_CUDA_TRY(cudaFuncSetAttribute(k_syrk<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)step_smem<T>()));
    return true;
  }();
  (void)attr;
  for (int J0 = 0; J0 < pmax; J0 += NB2) {
    const int jend = outer ? J0 + NB2 : INT_MAX;
    for (int j0 = J0; j0 < std::min(pmax, J0 + NB2); j0 += NB) {
      // active fronts, and those with rows below the block (sorted by p,
      // largest first)
      int nact = 0, nbelow = 0;
      while (nact < nfront && lead[nact].p > j0) ++nact;
      while (nbelow < nact && lead[nbelow].p > j0 + NB) ++nbelow;
      const int rest = std::max(0, lead[0].p - j0 - NB);
      const int ntile = ceil_div(rest, TILE);
      const int nctile = outer ? ceil_div(std::min(rest, jend - j0 - NB), TILE) : 0;
      const int grid = outer ? ntile * nctile : ntile * (ntile + 1) / 2;
      // algorithmic counts of this step (only while profiling)
      double pf = 0, pb = 0, sf = 0, sb = 0;
      if (prof_enabled()) {
        for (int f = 0; f < nact; ++f) {
          const double jb = std::min(NB, lead[f].p - j0);
          const double rest = lead[f].p - j0 - jb;
          const double cols = std::min<double>(rest, (double)std::min(jend, lead[f].p) - j0 - jb);
          pf += 2.0 * jb * jb * jb / 3.0 + rest * jb * jb;
          pb += sizeof(T) * (jb * jb + 2.0 * rest * jb);
          sf += (2.0 * rest - cols + 1.0) * cols * jb;
          sb += sizeof(T) * (rest * jb + (2.0 * rest - cols + 1.0) * cols);
        }
      }
      for (int f0 = 0; f0 < nact; f0 += MAX_GRID_Y) {
        const int nb = std::min(MAX_GRID_Y, nact - f0);
        ProfScope ps("chol_panel", st, pf, pb);
        k_chol_diag<T><<<nb, 256, chol_diag_smem<T>(), st>>>(d_lead + f0, Karena, Parena, j0,
                                                            d_flags,
                                                            growth_on ? (float)retry->growth : 0.f,
                                                            growth_on ? d_fflag + f0 : nullptr);
        HIF_CHECK_LAUNCH();
      }
      if (nbelow == 0) continue;
      if constexpr (sizeof(T) == 8) {
        if (f64tc) {
          std::vector<GemmOp> po(nbelow), uo(nbelow);
          for (int f = 0; f < nbelow; ++f) {
            const DFront& h = lead[f];
            const int ld = h.ld, r = h.p - j0 - NB;
            const int64_t a21 = h.K + j0 + NB + (int64_t)j0 * ld;
            po[f] = GemmOp{a21, h.P + j0 + (int64_t)j0 * ld, a21, r, NB, NB, ld, ld, ld, 0, 1, 1.f, 0.f,
                           0, KZ_B_UP, KB_DOWN, (int64_t)f * kstride + j0};
            uo[f] = GemmOp{a21, a21, a21 + (int64_t)NB * ld, r, r, NB, ld, ld, ld, 0, 1, -1.f, 1.f, 1, 0};
          }
          GemmOp* d_step = nullptr;
          HIF_CUDA_TRY(cudaMallocAsync(&d_step, sizeof(GemmOp) * 2 * nbelow, st));
          po.insert(po.end(), uo.begin(), uo.end());
          HIF_CUDA_TRY(cudaMemcpyAsync(d_step, po.data(), sizeof(GemmOp) * 2 * nbelow,
                                       cudaMemcpyHostToDevice, st));
          gemm_f64tc<double>(d_step, po.data(), nbelow, Karena, Parena, Karena, d_flags, st, "chol_panel_f64tc",
                             d_kexp);
          gemm_f64tc<double>(d_step + nbelow, uo.data(), nbelow, Karena, Karena, Karena, d_flags, st,
                     "chol_trailing_update_f64tc");
          HIF_CUDA_TRY(cudaFreeAsync(d_step, st));
          continue;
        }
      }
      for (int f0 = 0; f0 < nbelow; f0 += MAX_GRID_Y) {
        const int nb = std::min(MAX_GRID_Y, nbelow - f0);
        {
          ProfScope ps("chol_panel", st);
          k_panel<T><<<dim3(ntile, nb), 256, step_smem<T>(), st>>>(d_lead + f0, Karena, Parena, j0);
          HIF_CHECK_LAUNCH();
        }
        if (grid == 0) continue;
        ProfScope ps("chol_trailing_update", st, sf, sb);
        k_syrk<T><<<dim3(grid, nb), 256, step_smem<T>(), st>>>(d_lead + f0, Karena, j0,
                                                              outer ? jend : INT_MAX);
        HIF_CHECK_LAUNCH();
      }
    }
    if (!outer) continue;
    // A22 -= L21 L21^T for the fronts that extend past the outer block
    std::vector<GemmOp> uo;
    for (int f = 0; f < nfront && lead[f].p > jend; ++f) {
      const DFront& h = lead[f];
      const int64_t ld = h.ld;
      const int rest = h.p - jend;
      uo.push_back(GemmOp{h.K + jend + (int64_t)J0 * ld, h.K + jend + (int64_t)J0 * ld,
                          h.K + jend + (int64_t)jend * ld, rest, rest, NB2, (int)ld, (int)ld,
                          (int)ld, 0, 1, -1.f, 1.f, 1, 0});
    }
    if (uo.empty()) continue;
    GemmOp* d_uo = nullptr;
    HIF_CUDA_TRY(cudaMallocAsync(&d_uo, sizeof(GemmOp) * uo.size(), st));
    HIF_CUDA_TRY(cudaMemcpyAsync(d_uo, uo.data(), sizeof(GemmOp) * uo.size(),
                                 cudaMemcpyHostToDevice, st));
    bool done = false;
    if constexpr (std::is_same<T, float>::value) {
      if (tensor_cores) {
        gemm_tc(d_uo, uo.data(), (int)uo.size(), Karena, Karena, Karena, d_flags, st,
                "chol_block_update_tc");
        done = true;
      }
    }
    if (!done)
      gemm_fma_or_f64tc<T>(d_uo, uo.data(), (int)uo.size(), Karena, Karena, Karena, d_flags,
                           tensor_cores, st, "chol_block_update", "chol_block_update_f64tc");
    HIF_CUDA_TRY(cudaFreeAsync(d_uo, st));
  }
  HIF_CUDA_TRY(cudaFreeAsync(d_lead, st));
  // flagged fronts: redone in FP64 now; the others go on in FP32
  std::vector<DFront> keep;
  DFront* d_keep = nullptr;
  if (growth_on) {
    std::vector<int> hf(nfront), bad;
    HIF_CUDA_TRY(cudaMemcpyAsync(hf.data(), d_fflag, sizeof(int) * nfront, cudaMemcpyDeviceToHost, st));
    HIF_CUDA_TRY(cudaStreamSynchronize(st));
    for (int f = 0; f < nfront; ++f) {
      if (hf[f]) bad.push_back(f);
      else keep.push_back(h_fronts[f]);
    }
    if (!bad.empty()) {
      if constexpr (std::is_same<T, float>::value)
        retry_fronts_fp64(bad, h_fronts, soff, Karena, Parena, snap, d_flags, retry->tensor_cores, st);
      if (retry->retried) *retry->retried += (int64_t)bad.size();
      if (!keep.empty()) {
        HIF_CUDA_TRY(cudaMallocAsync(&d_keep, sizeof(DFront) * keep.size(), st));
        HIF_CUDA_TRY(cudaMemcpyAsync(d_keep, keep.data(), sizeof(DFront) * keep.size(),
                                     cudaMemcpyHostToDevice, st));
      }
      d_fronts = d_keep;
      h_fronts = keep.data();
      nfront = (int)keep.size();
    }
    HIF_CUDA_TRY(cudaFreeAsync(d_soff, st));
    snap_b.release();
    HIF_CUDA_TRY(cudaFreeAsync(d_fflag, st));
    if (nfront == 0) return;
  }
  finish_fronts(d_fronts, h_fronts, nfront, Karena, Parena, d_flags, tensor_cores, st, d_kexp, kstride);
  if (d_keep) HIF_CUDA_TRY(cudaFreeAsync(d_keep, st));
}

// Steps 2-4 of the partial Cholesky once the leading blocks hold L.  d_kexp: the
// exponents of the eliminated DOFs' scales, kstride per front (FP64 on tensor cores).
template <typename T>
void finish_fronts(const DFront* d_fronts, const DFront* h_fronts, int nfront, T* Karena,
                   T* Parena, int* d_flags, bool tensor_cores, cudaStream_t st, const int* d_kexp,
                   int kstride) {
  const int pmax = h_fronts[0].p;
  // 2. Linv = L^{-1}: the diagonal blocks are inverted already; merge
  //    neighbouring inverted blocks pairwise up a binary tree of widths
  //    s = NB, 2 NB, 4 NB, ...:  inv([A 0; B C]) = [A^-1 0; -C^-1 B A^-1  C^-1]
  //    (two batched products per width: T = B A^-1, then -C^-1 T)
  for (int s = NB; s < pmax; s *= 2) {
    std::vector<GemmOp> tops, rops;
    int64_t scr = 0;
    for (int f = 0; f < nfront && h_fronts[f].p > s; ++f) {
      const DFront& h = h_fronts[f];
      const int ld = h.ld;
      for (int i0 = 0; i0 + s < h.p; i0 += 2 * s) {
        const int rs = std::min(2 * s, h.p - i0) - s;   // rows of the right part
        const int64_t boff = (i0 + s) + (int64_t)i0 * ld;
        const int64_t aoff = i0 + (int64_t)i0 * ld;
        const int64_t coff = (i0 + s) + (int64_t)(i0 + s) * ld;
        tops.push_back(GemmOp{h.K + boff, h.P + aoff, scr, rs, s, s, ld, ld, rs, 0, 0, 1.f, 0.f, 0, KZ_B_LOW,
                              KB_NONE, 0});
        rops.push_back(GemmOp{h.P + coff, scr, h.P + boff, rs, s, rs, ld, rs, ld, 0, 0, -1.f, 0.f, 0, KZ_A_LOW,
                              KB_UP, (int64_t)f * kstride + i0 + s});
        scr += (int64_t)rs * s;
      }
    }
    if (tops.empty()) break;
    const size_t cnt = tops.size();
    GemmOp* d_ops = nullptr;
    DevBuf scr_b;
    HIF_CUDA_TRY(cudaMallocAsync(&d_ops, sizeof(GemmOp) * 2 * cnt, st));
    T* d_scr = scr_b.scratch<T>(scr, st);
    HIF_CUDA_TRY(cudaMemcpyAsync(d_ops, tops.data(), sizeof(GemmOp) * cnt, cudaMemcpyHostToDevice, st));
    HIF_CUDA_TRY(cudaMemcpyAsync(d_ops + cnt, rops.data(), sizeof(GemmOp) * cnt,
                                 cudaMemcpyHostToDevice, st));
    auto gemm = [&](const GemmOp* dop, const GemmOp* hop, const T* Ab, const T* Bb, T* Cb) {
      if constexpr (std::is_same<T, float>::value) {
        if (tensor_cores && s >= 128) {
          gemm_tc(dop, hop, (int)cnt, Ab, Bb, Cb, d_flags, st, "trtri_merge_tc");
          return;
        }
      }
      gemm_fma_or_f64tc<T>(dop, hop, (int)cnt, Ab, Bb, Cb, d_flags, tensor_cores, st, "trtri_merge",
                           "trtri_merge_f64tc", d_kexp);
    };
    gemm(d_ops, tops.data(), Karena, Parena, d_scr);
    gemm(d_ops + cnt, rops.data(), Parena, d_scr, Parena);
    HIF_CUDA_TRY(cudaFreeAsync(d_ops, st));
  }
  // 3. X^T = A_NI L^{-T} (into the panel below Linv) and 4. the Schur
  //    complement A_NN -= X^T X (lower tiles), each one deep product per front
  std::vector<GemmOp> xo, so;
  int maxrows = 0;
  for (int f = 0; f < nfront; ++f) {
    const DFront& h = h_fronts[f];
    const int nb = h.n - h.p;
    if (nb <= 0 || h.p <= 0) continue;
    const int ld = h.ld;
    GemmOp x{h.K + h.p, h.P, h.P + h.p, nb, h.p, h.p, ld, ld, ld, 0, 1, 1.f, 0.f, 0, KZ_B_UP,
             KB_DOWN, (int64_t)f * kstride};
    GemmOp s{h.P + h.p, h.P + h.p, h.K + h.p + (int64_t)h.p * ld, nb, nb, h.p, ld, ld, ld, 0, 1,
             -1.f, 1.f, 1, 0};
    xo.push_back(x);
    so.push_back(s);
    maxrows = std::max(maxrows, nb);
  }
  if (!xo.empty()) {
    GemmOp* d_ops = nullptr;
    const size_t cnt = xo.size();
    HIF_CUDA_TRY(cudaMallocAsync(&d_ops, sizeof(GemmOp) * 2 * cnt, st));
    HIF_CUDA_TRY(cudaMemcpyAsync(d_ops, xo.data(), sizeof(GemmOp) * cnt, cudaMemcpyHostToDevice, st));
    HIF_CUDA_TRY(cudaMemcpyAsync(d_ops + cnt, so.data(), sizeof(GemmOp) * cnt,
                                 cudaMemcpyHostToDevice, st));
    auto gemm = [&](const GemmOp* dop, const GemmOp* hop, const T* Ab, const T* Bb, T* Cb) {
      if constexpr (std::is_same<T, float>::value) {
        if (tensor_cores && maxrows >= TC_MIN_ROWS) {
          gemm_tc(dop, hop, (int)cnt, Ab, Bb, Cb, d_flags, st);
          return;
        }
      }
      gemm_fma_or_f64tc<T>(dop, hop, (int)cnt, Ab, Bb, Cb, d_flags, tensor_cores, st, "gemm_batched",
                           "gemm_f64tc", d_kexp);
    };
    gemm(d_ops, xo.data(), Karena, Parena, Parena);
    gemm(d_ops + cnt, so.data(), Parena, Parena, Karena);
    HIF_CUDA_TRY(cudaFreeAsync(d_ops, st));
  }
}

void diag_exponents(const DFront* d_fronts, int nfront, const double* Karena, int* d_kexp, int stride,
                    cudaStream_t st) {
  if (nfront == 0) return;
  ProfScope ps("diag_exponents", st);
  k_diag_exponents<<<nfront, 128, 0, st>>>(d_fronts, Karena, d_kexp, stride);
  HIF_CHECK_LAUNCH();
}

template <typename T>
void gemm_batched(const GemmOp* d_ops, const GemmOp* h_ops, int nops, const T* Abase,
                  const T* Bbase, T* Cbase, cudaStream_t st, const char* name) {
  if (nops == 0) return;
  int mt = 1;
  for (int i = 0; i < nops; ++i)
    mt = std::max(mt, ceil_div(h_ops[i].m, TILE) * ceil_div(h_ops[i].n, TILE));
  for (int f0 = 0; f0 < nops; f0 += MAX_GRID_Y) {
    const int nb = std::min(MAX_GRID_Y, nops - f0);
    double fl = 0;
    if (prof_enabled())
      for (int i = f0; i < f0 + nb; ++i) fl += 2.0 * h_ops[i].m * (double)h_ops[i].n * h_ops[i].k * (h_ops[i].kzero ? 0.5 : 1.0);
    ProfScope ps(name, st, fl, 0.0);
    k_gemm<T><<<dim3(mt, nb), 256, 0, st>>>(d_ops + f0, Abase, Bbase, Cbase);
    HIF_CHECK_LAUNCH();
  }
}

#define HIF_INST(T)                                                                          \
  template void partial_cholesky<T>(const DFront*, const DFront*, int, T*, T*, int*, bool,  \
                                    cudaStream_t, const RetryOpts*);                         \
  template void gemm_batched<T>(const GemmOp*, const GemmOp*, int, const T*, const T*, T*,  \
                                cudaStream_t, const char*);
HIF_INST(float)
HIF_INST(double)
#undef HIF_INST

}  // namespace hif
