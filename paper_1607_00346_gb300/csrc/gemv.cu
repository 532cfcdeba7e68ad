// Batched mat-vecs of the apply sweeps: y = alpha op(M) x (+ y) for many
// small-to-large column-major matrices of the factor and 1-16 right-hand
// sides at once.
//
// What bounds them: each factor entry is read once per sweep and used in one
// multiply-add per right-hand side, so up to 16 FP32 columns they are bound by
// HBM; what has to be kept off the critical path is the latency of the loads
// (every warp keeps 16 or more 128-byte loads in flight), the loads of x (one
// per matrix entry and column if x is not shared) and the idle warps of uneven
// batches (sizes go from 27 x 27 to thousands within one sweep).
//
// Work is cut into tasks on the host, once per list (gemv_plan), so that a
// launch has no empty blocks:
//   * M x: a task is a 64-row tile of one matrix.  1, 2, 4 or 8 warps of a
//     256-thread CTA share it (by the tile's column count, 8 columns per
//     block, blocks dealt to the warps in turn), so a CTA holds 8, 4, 2 or 1
//     tiles; the warps' sums are added in warp order through shared memory.
//     x of a block goes through a warp-private corner of shared memory and is
//     read back as broadcasts.
//   * M^T x: a task is 32 columns of one matrix, eight for each warp of a
//     128-thread CTA; lanes stride the rows and share each x value between
//     the eight columns; a transposing butterfly adds the lanes.
// The order of every sum depends on the matrix shape only, so a column gets
// the same bits in any block of right-hand sides.
//
// Measured on a 128^3 FP32 factor (2.86e9 entries, 22.9 GB in the two sweeps),
// the mat-vecs of one apply: 1 column 3.9 ms (5.9 TB/s), 4 columns 5.0 ms, 16
// columns 8.7 ms; with one CTA per 128 rows or 8 columns and x read from L1 by
// every warp (blocks 16, 8, 4, 2, 1) they took 6.5 ms for 1 column and 37 ms
// for 16.  On a 64^3 FP64 factor an apply of 8 columns takes 7.7 ms, 7.2 ms of which
// are the multiply-adds at the FP64 rate.
#include <algorithm>
#include <vector>

#include "dense.cuh"

namespace hif {

namespace {

constexpr int GEMV_THREADS = 256;
constexpr int GEMV_WARPS = GEMV_THREADS / 32;
constexpr int GEMV_TR = 64;    // rows of an M x tile, two per lane
constexpr int GEMV_BC = 8;     // columns of a block of an M x tile
constexpr int GEMV_T_THREADS = 128;
constexpr int GEMV_CG = 8;     // columns of a warp of M^T x
constexpr int GEMV_CG_FINE = 2;   // the same in the fine form
constexpr int GEMV_TC = GEMV_CG * GEMV_T_THREADS / 32;   // columns of an M^T x task

// R consecutive values from shared memory, as 16-byte vectors where they fill one.
template <int R>
__device__ __forceinline__ void read_x(float (&t)[R], const float* p) {
  if constexpr (R >= 4) {
#pragma unroll
    for (int q = 0; q < R; q += 4) {
      const float4 a = *reinterpret_cast<const float4*>(p + q);
      t[q] = a.x;
      t[q + 1] = a.y;
      t[q + 2] = a.z;
      t[q + 3] = a.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < R; ++q) t[q] = p[q];
  }
}
template <int R>
__device__ __forceinline__ void read_x(double (&t)[R], const double* p) {
  if constexpr (R >= 2) {
#pragma unroll
    for (int q = 0; q < R; q += 2) {
      const double2 a = *reinterpret_cast<const double2*>(p + q);
      t[q] = a.x;
      t[q + 1] = a.y;
    }
  } else {
    t[0] = p[0];
  }
}

// ---- y = alpha M x (+ y) --------------------------------------------------------
// One tile by `ncls` warps, this one taking blocks cls, cls + ncls, ...; the
// caller's warps of one CTA all come here with the same ncls.  xs: this
// warp's GEMV_BC x R corner; red: the CTA's GEMV_WARPS x GEMV_TR x RQ sums.
template <typename T, int R>
__host__ __device__ constexpr int gemv_red_cols() {   // right-hand sides reduced per round
  return R < 4 ? R : 4;
}

// RL = 2: the whole tile, two rows per lane; RL = 1: its half `half`.
template <typename T, int R, int RL>
__device__ __forceinline__ void gemv_n_tile(const GemvList<T>& sg, bool valid, int ti, int half,
                                            int ncls, T* xs_all, T* red) {
  constexpr int TR = 32 * RL;
  constexpr int XN = (GEMV_BC * R + 31) / 32;   // x values a lane stages per block
  constexpr int RQ = gemv_red_cols<T, R>();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int cls = warp % ncls;
  T* xs = xs_all + warp * (GEMV_BC * R);
  GemvTask tk{0, 0};
  GemvOp o{};
  if (valid) {
    tk = sg.tasks[ti];
    o = sg.ops[tk.op];
  }
  const int r0 = tk.tile * GEMV_TR + 32 * half;
  const int rows = o.rows;
  const int cols = valid ? (o.tri ? min(o.cols, r0 + TR) : o.cols) : 0;
  const int nblk = (cols + GEMV_BC - 1) / GEMV_BC;
  const T* M = sg.M + o.M;
  const T* x = sg.w + o.x;
  const int64_t vs = sg.vs;
  const int nv = sg.nv;
  const bool rfull = r0 + TR <= rows;

  T acc[RL][R];
#pragma unroll
  for (int i = 0; i < RL; ++i)
#pragma unroll
    for (int q = 0; q < R; ++q) acc[i][q] = T(0);
  // a block's matrix entries and x values, in flight while the block before
  // it is multiplied
  constexpr bool AHEAD = sizeof(T) == 4 || R < 8;   // else the sums need the registers
  T m[RL][GEMV_BC], mn[RL][GEMV_BC], xv[XN], xn[XN];
  auto full = [&](int b) {   // no entry of the block is masked
    const int c0 = b * GEMV_BC;
    return rfull && c0 + GEMV_BC <= cols && (!o.tri || c0 + GEMV_BC <= r0 + 1);
  };
  auto load = [&](int b, T (&mm)[RL][GEMV_BC], T (&xx)[XN]) {
    const int c0 = b * GEMV_BC;
    const T* mc = M + (int64_t)c0 * o.ld;
    if (full(b)) {
#pragma unroll
      for (int c = 0; c < GEMV_BC; ++c)
#pragma unroll
        for (int i = 0; i < RL; ++i) mm[i][c] = mc[r0 + lane + 32 * i + (int64_t)c * o.ld];
    } else {
#pragma unroll
      for (int c = 0; c < GEMV_BC; ++c)
#pragma unroll
        for (int i = 0; i < RL; ++i) {
          const int r = r0 + lane + 32 * i;
          mm[i][c] = (c0 + c < cols && r < rows && (!o.tri || c0 + c <= r)) ? mc[r + (int64_t)c * o.ld]
                                                                           : T(0);
        }
    }
#pragma unroll
    for (int j = 0; j < XN; ++j) {
      const int e = lane + 32 * j, q = e / GEMV_BC, c = c0 + e % GEMV_BC;
      xx[j] = (q < nv && q < R && c < cols) ? x[q * vs + c] : T(0);
    }
  };
  if (AHEAD && cls < nblk) load(cls, m, xv);
  for (int b = cls; b < nblk; b += ncls) {
    if (!AHEAD) load(b, m, xv);
    else if (b + ncls < nblk) load(b + ncls, mn, xn);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < XN; ++j) {
      const int e = lane + 32 * j;
      if (e < GEMV_BC * R) xs[(e % GEMV_BC) * R + e / GEMV_BC] = xv[j];
    }
    __syncwarp();
    if (full(b)) {
#pragma unroll
      for (int c = 0; c < GEMV_BC; ++c) {
        T t[R];
        read_x<R>(t, xs + c * R);
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int i = 0; i < RL; ++i) acc[i][q] = fma(m[i][c], t[q], acc[i][q]);
      }
    } else {
      // a masked entry leaves its sum alone (x may be infinite there)
#pragma unroll
      for (int c = 0; c < GEMV_BC; ++c) {
        const int cc = b * GEMV_BC + c;
#pragma unroll
        for (int i = 0; i < RL; ++i) {
          if (cc >= cols || (o.tri && cc > r0 + lane + 32 * i)) continue;
#pragma unroll
          for (int q = 0; q < R; ++q) acc[i][q] = fma(m[i][c], xs[c * R + q], acc[i][q]);
        }
      }
    }
    if (AHEAD) {
#pragma unroll
      for (int c = 0; c < GEMV_BC; ++c)
#pragma unroll
        for (int i = 0; i < RL; ++i) m[i][c] = mn[i][c];
#pragma unroll
      for (int j = 0; j < XN; ++j) xv[j] = xn[j];
    }
  }
  const T al = (T)o.alpha;
  T* y = sg.w + o.y;
  if (ncls == 1) {
    if (!valid) return;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (q >= nv) continue;
#pragma unroll
      for (int i = 0; i < RL; ++i) {
        const int r = r0 + lane + 32 * i;
        if (r >= rows) continue;
        T* yp = y + q * vs + r;
        *yp = (o.beta_one ? *yp : T(0)) + al * acc[i][q];
      }
    }
    return;
  }
  // the warps' sums of each tile, added in warp order, RQ columns per round
  const int t0 = warp / ncls * ncls;               // first warp of this tile
  const int tid = (warp - t0) * 32 + lane;         // thread within the tile's warps
#pragma unroll
  for (int q0 = 0; q0 < R; q0 += RQ) {
    if (q0 >= nv) break;
#pragma unroll
    for (int q = 0; q < RQ; ++q)
#pragma unroll
      for (int i = 0; i < RL; ++i) red[(warp * RQ + q) * TR + lane + 32 * i] = acc[i][q0 + q];
    __syncthreads();
    if (valid)
      for (int e = tid; e < RQ * TR; e += ncls * 32) {
        const int q = e / TR, r = r0 + e % TR;
        T s = red[t0 * RQ * TR + e];
        for (int w = 1; w < ncls; ++w) s += red[(t0 + w) * RQ * TR + e];
        if (r < rows && q0 + q < nv) {
          T* yp = y + (q0 + q) * vs + r;
          *yp = (o.beta_one ? *yp : T(0)) + al * s;
        }
      }
    __syncthreads();
  }
}

template <typename T, int R, bool FINE>
__device__ __forceinline__ void gemv_n_cta(const GemvList<T>& sg, int b) {
  constexpr int RL = FINE ? 1 : 2;
  __shared__ __align__(16) T xs[GEMV_WARPS * GEMV_BC * R];
  __shared__ T red[GEMV_WARPS * gemv_red_cols<T, R>() * 32 * RL];
  const int warp = threadIdx.x / 32;
  const int half = FINE ? b % 2 : 0;
  if (FINE) b /= 2;
  // the list's tasks, those of 8 warps first, then 4, 2 and 1
  int ncls = 8, base = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int per = GEMV_WARPS / ncls;   // tiles per CTA
    const int nc = (sg.cnt[k] + per - 1) / per;
    if (b < nc || k == 3) {
      const int j = b * per + warp / ncls;
      gemv_n_tile<T, R, RL>(sg, j < sg.cnt[k], base + j, half, ncls, xs, red);
      return;
    }
    b -= nc;
    base += sg.cnt[k];
    ncls >>= 1;
  }
}

// One step of the butterfly over lanes S apart: the first N values of v are
// summed; a lane keeps half of them (which half: idx) while there are several.
template <typename T, int N, int S>
__device__ __forceinline__ void lane_sum(T* v, int lane, int& idx) {
  if constexpr (N > 1) {
    const bool up = (lane & S) != 0;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const T send = up ? v[i] : v[i + N / 2];
      const T keep = up ? v[i + N / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, S);
    }
    idx += up ? N / 2 : 0;
  } else {
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], S);
  }
  if constexpr (S > 1) lane_sum<T, (N > 1 ? N / 2 : 1), S / 2>(v, lane, idx);
}

// ---- y = alpha M^T x (+ y) -------------------------------------------------------
// One CTA of four warps, columns 32 tile .. 32 tile + 31, eight per warp;
// lanes stride the rows (from the 32-row step that holds the triangle's
// diagonal), and a transposing butterfly adds the lanes at the end.
//   * Up to 4 right-hand sides: x comes straight from L1, the loads of 2 row
//     steps (16 matrix entries per lane) in flight together.
//   * 8 and 16: x would be 8-16 loads per row step and the sums fill the
//     registers, so the CTA copies 128 rows (FP64: 64) of its 32 columns and
//     of x at a time to shared memory, asynchronously and one chunk ahead;
//     each value of x is then read once for eight columns.
// FP32, 16 columns, the T half of a 128^3 sweep (11.4 GB of factor): four
// columns per warp with x from L1 9.0 ms (waiting for x), eight with x in
// shared memory and the matrix in registers 6.5 ms (waiting for the matrix),
// this form 4.8 ms.
__device__ __forceinline__ void cp_async(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async(double* dst, const double* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 8 : 0) : "memory");
}

// Sums over the lanes and writes y of CG columns from c0 on.
template <typename T, int R, int CG>
__device__ __forceinline__ void gemv_t_finish(T (&v)[CG * R], const GemvOp& o, const GemvList<T>& sg,
                                              int c0) {
  constexpr int V = CG * R;
  const int lane = threadIdx.x % 32;
  // lane l ends with the values whose index has the bits of l (16, 8, ..) as
  // its leading bits
  int idx = 0;
  lane_sum<T, V, 16>(v, lane, idx);
  constexpr int KEEP = V > 32 ? V / 32 : 1;         // values left per lane
  constexpr int DUP = V < 32 ? 32 / V : 1;          // lanes that hold the same value
  if (lane % DUP) return;
  const T al = (T)o.alpha;
#pragma unroll
  for (int i = 0; i < KEEP; ++i) {
    const int c = c0 + (idx + i) / R, q = (idx + i) % R;
    if (c < o.cols && q < sg.nv) {
      T* yp = sg.w + o.y + q * sg.vs + c;
      *yp = (o.beta_one ? *yp : T(0)) + al * v[i];
    }
  }
}

template <typename T, int R, int CG>
__device__ __forceinline__ void gemv_t_few(const GemvList<T>& sg, int b) {
  constexpr int UN = 2 * GEMV_CG / CG;   // row steps in flight
  constexpr int SUB = GEMV_CG / CG;      // CTAs per task
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const GemvTask tk = sg.tasks[b / SUB];
  const GemvOp o = sg.ops[tk.op];
  const int c0 = tk.tile * GEMV_TC + (b % SUB * (GEMV_T_THREADS / 32) + warp) * CG;
  if (c0 >= o.cols) return;
  const int rows = o.rows;
  const int64_t vs = sg.vs, ld = o.ld;
  const int nv = sg.nv;
  const T* M = sg.M + o.M + (int64_t)c0 * ld;
  const T* x = sg.w + o.x;
  T v[CG * R];   // v[c R + q]
#pragma unroll
  for (int i = 0; i < CG * R; ++i) v[i] = T(0);
  auto masked = [&](int r) {
    if (r >= rows) return;
    T mm[CG];
#pragma unroll
    for (int c = 0; c < CG; ++c)
      mm[c] = (c0 + c < o.cols && (!o.tri || r >= c0 + c)) ? M[r + c * ld] : T(0);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const T xq = q < nv ? x[q * vs + r] : T(0);
#pragma unroll
      for (int c = 0; c < CG; ++c)
        if (!o.tri || r >= c0 + c) v[c * R + q] = fma(mm[c], xq, v[c * R + q]);
    }
  };
  int r = 0;
  if (o.tri) {
    r = c0 / 32 * 32;
    masked(r + lane);
    r += 32;
  }
  if (c0 + CG <= o.cols) {
    for (; r + 32 * UN <= rows; r += 32 * UN) {
      T mm[UN][CG], xq[UN][R];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
#pragma unroll
        for (int c = 0; c < CG; ++c) mm[u][c] = M[r + 32 * u + lane + c * ld];
#pragma unroll
        for (int q = 0; q < R; ++q) xq[u][q] = q < nv ? x[q * vs + r + 32 * u + lane] : T(0);
      }
#pragma unroll
      for (int u = 0; u < UN; ++u)
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int c = 0; c < CG; ++c) v[c * R + q] = fma(mm[u][c], xq[u][q], v[c * R + q]);
    }
  }
  for (; r < rows; r += 32) masked(r + lane);
  gemv_t_finish<T, R, CG>(v, o, sg, c0);
}

// 8 or 16 right-hand sides.
template <typename T, int R, int CG>
__device__ __forceinline__ void gemv_t_many(const GemvList<T>& sg, int b) {
  constexpr int SUB = GEMV_CG / CG;                         // CTAs per task
  constexpr int TC = GEMV_TC / SUB;                         // columns of the CTA
  constexpr int CH = GEMV_T_THREADS * 4 / (int)sizeof(T);   // rows per chunk
  constexpr int STEPS = CH / 32;
  constexpr int CPR = GEMV_T_THREADS / CH;                  // columns copied side by side
  __shared__ T ms[2][TC][CH];
  __shared__ T xs[2][R][CH];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const GemvTask tk = sg.tasks[b / SUB];
  const GemvOp o = sg.ops[tk.op];
  const int ct = tk.tile * GEMV_TC + b % SUB * TC, c0 = ct + warp * CG;
  if (ct >= o.cols) return;
  const int rows = o.rows;
  const int64_t vs = sg.vs, ld = o.ld;
  const T* M = sg.M + o.M + (int64_t)ct * ld;
  const int rbeg = o.tri ? tk.tile * GEMV_TC : 0;   // GEMV_TC = 32: the diagonal's row step
  const int nchunk = rows > rbeg ? (rows - rbeg + CH - 1) / CH : 0;
  const int te = threadIdx.x % CH, tc = threadIdx.x / CH;
  const int nv = sg.nv;
  const T* x = sg.w + o.x;
  // chunk k of the matrix columns and of x, copied asynchronously; entries
  // outside the matrix or the triangle are zero
  auto stage = [&](int k) {
    if (k < nchunk) {
      const int r = rbeg + k * CH + te;
      const bool in = r < rows;
      if (ct + TC <= o.cols && (k + 1) * CH <= rows - rbeg && (!o.tri || k > 0)) {
        const T* m = M + r + tc * ld;
#pragma unroll
        for (int c = 0; c < TC; c += CPR) cp_async(&ms[k & 1][c + tc][te], m + c * ld, true);
      } else {
#pragma unroll
        for (int c = 0; c < TC; c += CPR) {
          const bool ok = in && ct + c + tc < o.cols && (!o.tri || r >= ct + c + tc);
          cp_async(&ms[k & 1][c + tc][te], ok ? M + r + (c + tc) * ld : x, ok);
        }
      }
#pragma unroll
      for (int q = 0; q < R; q += CPR) {
        const bool ok = in && q + tc < nv;
        cp_async(&xs[k & 1][q + tc][te], ok ? x + (q + tc) * vs + r : x, ok);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  T v[CG * R];
#pragma unroll
  for (int i = 0; i < CG * R; ++i) v[i] = T(0);
  stage(0);
  for (int k = 0; k < nchunk; ++k) {
    stage(k + 1);
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    const T(*mk)[CH] = &ms[k & 1][warp * CG];
    const T(*xk)[CH] = xs[k & 1];
#pragma unroll
    for (int s = 0; s < STEPS; ++s) {
      T m[CG];
#pragma unroll
      for (int c = 0; c < CG; ++c) m[c] = mk[c][32 * s + lane];
      if (s == 0 && k == 0 && o.tri) {
        // a masked entry leaves its sum alone (x may be infinite there)
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const T xq = xk[q][lane];
#pragma unroll
          for (int c = 0; c < CG; ++c)
            if (rbeg + lane >= c0 + c) v[c * R + q] = fma(m[c], xq, v[c * R + q]);
        }
      } else {
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const T xq = xk[q][32 * s + lane];
#pragma unroll
          for (int c = 0; c < CG; ++c) v[c * R + q] = fma(m[c], xq, v[c * R + q]);
        }
      }
    }
    __syncthreads();   // the chunk's buffers are free for chunk k + 2
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  gemv_t_finish<T, R, CG>(v, o, sg, c0);
}

template <typename T, int R, bool FINE>
__device__ __forceinline__ void gemv_t_cta(const GemvList<T>& sg, int b) {
  constexpr int CG = FINE ? GEMV_CG_FINE : GEMV_CG;
  if constexpr (R >= 8) gemv_t_many<T, R, CG>(sg, b);
  else gemv_t_few<T, R, CG>(sg, b);
}

// M x, FP32 up to 4 columns: three CTAs per SM keep 24 warps of loads in
// flight; 8 and 16 columns (and FP64) need the registers for their sums.
// M^T x, 8 and 16 columns: the sums fill the registers, two or three CTAs of
// four warps keep a chunk each in flight.
template <int TRANS>
constexpr int gemv_threads() { return TRANS ? GEMV_T_THREADS : GEMV_THREADS; }
template <int TRANS>   // fine blocks per coarse block
__host__ __device__ constexpr int gemv_finer() { return TRANS ? GEMV_CG / GEMV_CG_FINE : 2; }
template <typename T, int R, int TRANS>
constexpr int gemv_ctas_per_sm() {
  if (TRANS) return R >= 8 ? (sizeof(T) == 8 ? 2 : R == 16 ? 3 : 4) : sizeof(T) == 4 ? 6 : R < 4 ? 5 : 4;
  return sizeof(T) == 4 ? (R >= 8 ? 2 : 3) : 2;
}

template <typename T, int R, int TRANS, bool FINE>
__global__ void __launch_bounds__(gemv_threads<TRANS>(), (gemv_ctas_per_sm<T, R, TRANS>()))
    k_gemv(const GemvList<T> sg) {
  if constexpr (TRANS) gemv_t_cta<T, R, FINE>(sg, blockIdx.x);
  else gemv_n_cta<T, R, FINE>(sg, blockIdx.x);
}

// A launch with fewer coarse blocks than this takes the fine form: half the
// rows per CTA (M x) or a quarter of the columns (M^T x), the same sums.  Two
// blocks per SM: below that SMs idle while others, in FP64 above all, work
// through their tile (20^3 FP64, 10 columns: 7.6 ms a solve with the coarse
// form alone, 4.9 ms with one column per warp).
int gemv_fine_below() {
  static const int n = [] {
    int dev = 0, count = 0;
    HIF_CUDA_TRY(cudaGetDevice(&dev));
    HIF_CUDA_TRY(cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev));
    return 2 * count;
  }();
  return n;
}

template <typename T, int R, int TRANS>
void launch_gemv(const GemvList<T>& sg, cudaStream_t st) {
  const int ctas = gemv_ctas(sg.cnt);
  if (ctas < gemv_fine_below())
    k_gemv<T, R, TRANS, true><<<ctas * gemv_finer<TRANS>(), gemv_threads<TRANS>(), 0, st>>>(sg);
  else
    k_gemv<T, R, TRANS, false><<<ctas, gemv_threads<TRANS>(), 0, st>>>(sg);
  HIF_CHECK_LAUNCH();
}

}  // namespace

// Warps per tile of M x: enough blocks of 8 columns for each warp to keep a
// second block in flight, one warp for tiles of up to 4 blocks.
void gemv_plan(const GemvOp* ops, int nops, int trans, std::vector<GemvTask>& tasks, int (&cnt)[4]) {
  tasks.clear();
  for (int k = 0; k < 4; ++k) cnt[k] = 0;
  if (trans) {
    for (int i = 0; i < nops; ++i)
      for (int t = 0; (int64_t)t * GEMV_TC < ops[i].cols; ++t) tasks.push_back(GemvTask{i, t});
    cnt[0] = (int)tasks.size();
    return;
  }
  std::vector<GemvTask> by[4];
  for (int i = 0; i < nops; ++i)
    for (int t = 0; (int64_t)t * GEMV_TR < ops[i].rows; ++t) {
      const int c = ops[i].tri ? (int)std::min<int64_t>(ops[i].cols, ((int64_t)t + 1) * GEMV_TR) : ops[i].cols;
      by[c > 512 ? 0 : c > 128 ? 1 : c > 32 ? 2 : 3].push_back(GemvTask{i, t});
    }
  for (int k = 0; k < 4; ++k) {
    cnt[k] = (int)by[k].size();
    tasks.insert(tasks.end(), by[k].begin(), by[k].end());
  }
}

int gemv_ctas(const int (&cnt)[4]) {
  return cnt[0] + ceil_div(cnt[1], 2) + ceil_div(cnt[2], 4) + ceil_div(cnt[3], 8);
}

int gemv_block(int left, size_t word) {
  if (word == 8) return left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
  return left > 8 ? 16 : left > 4 ? 8 : left > 2 ? 4 : left;
}

template <typename T>
void gemv_batched(const GemvOp* h_ops, int nops, const GemvList<T>& list, int trans, int nrhs,
                  cudaStream_t st) {
  if (nops == 0 || gemv_ctas(list.cnt) == 0) return;
  for (int q0 = 0; q0 < nrhs;) {
    const int R = gemv_block(nrhs - q0, sizeof(T));
    GemvList<T> sg = list;
    sg.w = list.w + (int64_t)q0 * list.vs;
    sg.nv = std::min(R, nrhs - q0);
    double by = 0, fl = 0;
    if (prof_enabled()) {
      for (int i = 0; i < nops; ++i) {
        const GemvOp& o = h_ops[i];
        const double ent = o.tri ? 0.5 * (double)o.cols * (o.cols + 1) : (double)o.rows * o.cols;
        by += sizeof(T) * (ent + (double)sg.nv * (o.rows + o.cols) * (o.beta_one ? 1.5 : 1.0));
        fl += 2.0 * ent * sg.nv;
      }
    }
    ProfScope ps(trans ? "apply_gemv_t" : "apply_gemv_n", st, fl, by);
    if constexpr (sizeof(T) == 4)
      if (R == 16) trans ? launch_gemv<T, 16, 1>(sg, st) : launch_gemv<T, 16, 0>(sg, st);
    switch (R) {
      case 16: break;   // FP32 only (gemv_block)
      case 8: trans ? launch_gemv<T, 8, 1>(sg, st) : launch_gemv<T, 8, 0>(sg, st); break;
      case 4: trans ? launch_gemv<T, 4, 1>(sg, st) : launch_gemv<T, 4, 0>(sg, st); break;
      case 2: trans ? launch_gemv<T, 2, 1>(sg, st) : launch_gemv<T, 2, 0>(sg, st); break;
      default: trans ? launch_gemv<T, 1, 1>(sg, st) : launch_gemv<T, 1, 0>(sg, st);
    }
    q0 += sg.nv;
  }
}

#define HIF_INST(T) \
  template void gemv_batched<T>(const GemvOp*, int, const GemvList<T>&, int, int, cudaStream_t);
HIF_INST(float)
HIF_INST(double)
#undef HIF_INST

}  // namespace hif
