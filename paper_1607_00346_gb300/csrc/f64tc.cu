// Batched FP64 matrix products on the tensor cores.
//
// What bounds an FP64 product here is the FP64 unit: 2 multiply-adds per clock
// and SM, 1.06 TFLOP/s on the whole chip, so a single 64 x 64 x 64 tile takes
// 66 us and the products of a 64^3 FP64 factorization took 60% of its time.
// The BF16 tensor cores run 2300 times faster, and integers of 8 bits multiply
// and add in them without rounding; so each operand is split into eight 8-bit
// slices (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012):
//
//   x = 2^(s - 63) X,  X = sum_{i < 8} a_i 256^(7 - i),  |a_i| <= 128,
//
// with s per row of op(A) and per column of op(B) such that |x| < (1 - 2^-7) 2^s (room
// for the carry into a_0): X is x in fixed point, 62 to 63 bits below the largest entry
// of its row.  Before that, k is balanced: column k of op(A) is scaled by 2^t_k and row
// k of op(B) by 2^-t_k, so that an operand's own scale in k hides none of its entries.
// Write a front as D A^ D with D^2 its diagonal.  Then L = D L^ has no scale in its
// columns; A_NI = D A^ D and L^-T = D^-1 L^^-T have opposite ones in k, as have C^-1
// and T in the second product of a triangular merge and A_FF and T in the skeleton
// products.  So t_k is the exponent of D_k there (KB_DOWN, KB_UP; diag_exponents) and 0
// in the merges' first product (KB_NONE); only the products of the row reduction take
// half the difference of the operands' largest exponents (KB_MAX).  That was the rule
// of all products at first, but the largest entry of column k of A_NI says which DOFs
// k is coupled to, not how large k is: coefficients over six decades in blocks, layers
// or a ramp lost 30 to 200 times the FMA form's error (x of O(1) everywhere, 2-norm).
//
// The product is sum_t 256^(14 - t) D_t, D_t = sum_{i + j = t} sum_k a_i b_j; the 36
// products with t < 8 are formed in eight FP32 accumulators.  (Left out are seven
// products a_i b_j per k with t = 8, and smaller ones: at most 2^-61 of 2^s 2^s' per k,
// 2^-64 in the mean square.  With X one bit lower in a_0 they were four times as large,
// and holes of 10^3.5 doubled the FMA form's largest error.)  |D_t| <= 8 * 128 * 2^14 =
// 2^24 over 128 k, which FP32 holds exactly; then they are added to 128-bit integers
// (two 64-bit halves per entry), and each entry is rounded to double once at the end.
// An FMA loop rounds at every k; this sum is exact up to the split.
//
// Three launches per batch (four with KB_MAX, whose t_k k_f64_kmax finds): k_f64_exps
// finds s per row, k_f64_slice writes the slices in the layout the tensor core reads (64 rows
// x 16 k per block, all eight slices together: 16 KB), k_gemm_f64tc copies blocks
// to shared memory with bulk copies and multiplies.  An operand used on both
// sides (A A^T) is split once; if all products of a batch are such and have at most
// 64 k (the Cholesky updates), k_f64_slice_rows finds s and writes the slices with
// one read.
//
// Measured (all launches, FMA form in brackets): one 64^3 product 34 (76) us, 512 of
// them 108 (274) us, A A^T 28 (74) and 81 (270) us; one 256^3 48 (287) us, one 1024^3
// 0.106 (2.14) ms, one 2048^3 0.63 (14.5) ms = 27 TFLOP/s (by maxima, four launches,
// 0.66 ms).  Error against extended precision: 2e-17 to 6e-17 in norm.  For the solve
// error of a factorization see SLICE_SPAN in hif.cu.
//
// k_gemm_f64tc: one 128 x 64 tile per CTA; the eight accumulators fill the 512
// columns of tensor memory, four stages of 48 KB the shared memory.  Per 16 k one
// thread issues 12 instructions (M 128, N 64 to 256, K 16: a slice of A times
// up to four neighbouring slices of B, whose products go to neighbouring
// accumulators), and a warp copies the block three ahead; per 128 k the warps
// read the accumulators back.  A small tile is a chain of latencies (table,
// exponents, copies, products, C): exponents are read while tensor memory is
// allocated, C is copied to shared memory during the last read-back, and 512 threads of
// 16 columns each round the sums (256 of 32: 22.3 instead of 17.5 us for one 64^3
// tile; large products 3% slower).  This kernel alone: 1520 tiles of 64 k 166 us, 256^3
// 29 us, 1024^3 81, 2048^3 570, where the copies from L2 (6.4 TB/s) are the bound.
// With that and the one-pass slices a 64^3 FP64 factorization and solve went from 203 to
// 194 ms, a 32^3 periodic one from 45.3 to 42.5 ms.
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "dense.cuh"
#include "tcgen05.cuh"

namespace hif {

namespace {

constexpr int NSL = 8;             // slices per operand, and accumulators
// slices multiplied: all for FP64 operands.  FP32 operands (24 bits an entry) leave out
// the last slice of each and the products with t = 7: their rows are then rounded 55
// bits below the largest entry, which is as far as an FP64 FMA loop carries the sum.
// (28 instead of 36 products; Gram matrices of a 128^3 FP32 factorization 60.8 -> 56.0
// ms, of 96^3 13.4 -> 12.4 ms.)
template <typename S>
constexpr int slices_used() { return sizeof(S) == 4 ? NSL - 1 : NSL; }
constexpr int BR = 64;             // rows of a block of slices
constexpr int KC = 16;             // k of a block
constexpr int SLICE = BR * KC * 2;         // bytes of one slice of a block (2 KB)
constexpr int BLK = NSL * SLICE;           // bytes of a block (16 KB)
constexpr int TM = 128, TN = 64;           // output tile
constexpr int NST = 4;                     // shared-memory stages
constexpr int STAGE = 3 * BLK;             // two blocks of A, one of B
constexpr int GROUP = 8;                   // blocks (128 k) per exact accumulation
constexpr int THREADS = 512;
constexpr int CW = TN * 128 / THREADS;     // columns of a thread: four warps share a row of lanes
constexpr int NOT_FINITE = INT32_MAX;      // exponent of a row with inf or NaN
constexpr long long WAIT_LIMIT = 20000000;  // mbarrier polls before giving up
constexpr size_t WORK_LIMIT = (size_t)1 << 30;   // slices held at once, if several products

// 64 rows (row0 ..) of an operand: element (r, k) at src + r + k ld, or
// src + k + r ld (kcont).
struct SliceBlk {
  int64_t src;
  int64_t dst;       // index of its first 16 KB block in the work space
  int64_t kx;        // KB_MAX: index of the largest magnitudes of its product's
                     // columns of op(A), then rows of op(B) (k each); KB_DOWN and
                     // KB_UP: index of its exponents (GemmOp::ks)
  int ld, rows, k;
  int kcont, isB;
  int kbal;
};

struct Tile {
  int op, rb, cb;    // product, first row and column
  int ablk, bblk;    // first block row of A (two if the product has the rows), of B
};

// Largest magnitude over a block's rows for each k, as the upper word of its
// double (kx zeroed before; gridDim.y CTAs share the block's k).
template <typename S>
__global__ void __launch_bounds__(256) k_f64_kmax(const SliceBlk* __restrict__ blks,
                                                  const S* __restrict__ Ab,
                                                  const S* __restrict__ Bb, int* kx) {
  const SliceBlk b = blks[blockIdx.x];
  if (b.kbal != KB_MAX) return;
  const S* X = (b.isB ? Bb : Ab) + b.src;
  int* out = kx + b.kx + (b.isB ? b.k : 0);
  const int k0 = (int)((int64_t)b.k * blockIdx.y / gridDim.y);
  const int k1 = (int)((int64_t)b.k * (blockIdx.y + 1) / gridDim.y);
  if (b.kcont) {
    for (int k = k0 + threadIdx.x; k < k1; k += 256) {
      int m = 0;
#pragma unroll 8
      for (int r = 0; r < b.rows; ++r)
        m = max(m, __double2hiint((double)X[(int64_t)r * b.ld + k]) & 0x7fffffff);
      atomicMax(&out[k], m);
    }
  } else {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
#pragma unroll 4
    for (int k = k0 + warp; k < k1; k += 8) {
      int m = 0;
      for (int r = lane; r < b.rows; r += 32)
        m = max(m, __double2hiint((double)X[r + (int64_t)k * b.ld]) & 0x7fffffff);
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) atomicMax(&out[k], m);
    }
  }
}

// The exponent added to this operand's entries at k.  (BAL: some product of the batch is
// balanced; the loads and branches cost the Gram matrices, which are not, 3%.)
template <bool BAL>
__device__ __forceinline__ int balance(const SliceBlk& b, const int* kx,
                                       const int* __restrict__ kexp, int k) {
  if (!BAL || b.kbal == KB_NONE) return 0;
  if (b.kbal != KB_MAX) {
    const int e = kexp[b.kx + k];
    return (b.kbal == KB_UP) == (b.isB == 0) ? e : -e;
  }
  const int ea = kx[b.kx + k] >> 20, eb = kx[b.kx + b.k + k] >> 20;
  if (ea == 0 || eb == 0 || ea == 0x7ff || eb == 0x7ff) return 0;
  const int t = (eb - ea) >> 1;
  return b.isB ? -t : t;
}

// Largest balanced exponent of each row, biased by ROW_BIAS on top of the
// double's own bias so that a zero row is 0 (exps zeroed before; gridDim.y CTAs
// share the block's k).  Entries within 2^-6 of the next power of two count as that.
constexpr int ROW_BIAS = 4096;
constexpr int ROUND_UP = 1 << 14;   // 2^-6 of the upper word's mantissa
__device__ __forceinline__ int entry_exp(double x, int t) {
  const int h = __double2hiint(x) & 0x7fffffff, e = h >> 20;
  if (e == 0x7ff) return NOT_FINITE;
  if (h == 0 && __double2loint(x) == 0) return 0;
  return max((h + ROUND_UP) >> 20, 1) + t + ROW_BIAS;
}
template <typename S, bool BAL>
__global__ void __launch_bounds__(256) k_f64_exps(const SliceBlk* __restrict__ blks,
                                                  const S* __restrict__ Ab,
                                                  const S* __restrict__ Bb,
                                                  const int* __restrict__ kx,
                                                  const int* __restrict__ kexp, int* exps) {
  const SliceBlk b = blks[blockIdx.x];
  const S* X = (b.isB ? Bb : Ab) + b.src;
  const int k0 = (int)((int64_t)b.k * blockIdx.y / gridDim.y);
  const int k1 = (int)((int64_t)b.k * (blockIdx.y + 1) / gridDim.y);
  int* out = exps + (int64_t)blockIdx.x * BR;
  if (b.kcont) {
    // one warp per row, lanes along k
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int r = warp; r < b.rows; r += 8) {
      int m = 0;
#pragma unroll 4
      for (int k = k0 + lane; k < k1; k += 32)
        m = max(m, entry_exp(X[(int64_t)r * b.ld + k], balance<BAL>(b, kx, kexp, k)));
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) atomicMax(&out[r], m);
    }
  } else {
    const int r = threadIdx.x % BR;
    if (r >= b.rows) return;
    int m = 0;
#pragma unroll 8
    for (int k = k0 + threadIdx.x / BR; k < k1; k += 256 / BR)
      m = max(m, entry_exp(X[r + (int64_t)k * b.ld], balance<BAL>(b, kx, kexp, k)));
    atomicMax(&out[r], m);
  }
}

// s of a row, as a biased exponent: |x| < (1 - 2^-7) 2^(s - 1023) for all its entries
__device__ __forceinline__ int row_exp(int v) {
  return v == NOT_FINITE ? NOT_FINITE : v == 0 ? 1 : v - ROW_BIAS + 1;
}

// x in fixed point, 63 bits below 2^s (s: row_exp)
__device__ __forceinline__ int64_t fixed63(double x, int s) {
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  const int e = (int)(u >> 52) & 0x7ff;
  uint64_t m = u & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int sh = (e ? e : 1) - s + 11;   // at most 10
  uint64_t v;
  if (sh >= 0) v = m << sh;
  else if (sh > -55) v = (m + (1ull << (-sh - 1))) >> -sh;
  else v = 0;
  return (int64_t)u < 0 ? -(int64_t)v : (int64_t)v;
}

// Eight consecutive k (group g) of row r -> 16 bytes of each slice of a block.
__device__ __forceinline__ void write_slices(const double (&x)[8], int s, const int (&t)[8],
                                             unsigned char* blk, int r, int g) {
  // adding 128 to every digit but the first makes the bytes of the sum the
  // digits + 128; a byte put into the low mantissa of 2^23 and taken back
  // gives the digit as a float, whose upper half is its BF16
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint64_t y = (uint64_t)(s == NOT_FINITE ? 0 : fixed63(x[j], s - t[j])) + 0x8080808080808080ull;
    lo[j] = (uint32_t)y;
    hi[j] = (uint32_t)(y >> 32);
  }
  unsigned char* out = blk + (r / 8) * 256 + (g % 2) * 128 + (r % 8) * 16;
#pragma unroll
  for (int i = 0; i < NSL; ++i) {
    const uint32_t sel = 0x7440u | (uint32_t)((NSL - 1 - i) & 3);
    uint32_t d[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const uint32_t w0 = i < 4 ? hi[2 * h] : lo[2 * h], w1 = i < 4 ? hi[2 * h + 1] : lo[2 * h + 1];
      const float f0 = __uint_as_float(__byte_perm(w0, 0x4b000000u, sel)) - 8388736.0f;
      const float f1 = __uint_as_float(__byte_perm(w1, 0x4b000000u, sel)) - 8388736.0f;
      d[h] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
    }
    *reinterpret_cast<uint4*>(out + i * SLICE) = make_uint4(d[0], d[1], d[2], d[3]);
  }
}

// One thread: eight consecutive k of one row at a time.
template <typename S, bool BAL>
__global__ void __launch_bounds__(256) k_f64_slice(const SliceBlk* __restrict__ blks,
                                                   const S* __restrict__ Ab,
                                                   const S* __restrict__ Bb,
                                                   const int* __restrict__ kx,
                                                   const int* __restrict__ kexp,
                                                   const int* __restrict__ exps, unsigned char* W) {
  const SliceBlk b = blks[blockIdx.x];
  const S* X = (b.isB ? Bb : Ab) + b.src;
  // a warp covers 8 rows x 4 groups of 8 k: 512 contiguous bytes of two blocks
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int r = warp * 8 + lane % 8, kg = lane / 8;
  const int s = row_exp(exps[(int64_t)blockIdx.x * BR + r]);
  const int nkg = (b.k + KC - 1) / KC * 2;   // groups of 8 k, padded to whole blocks
  for (int g = blockIdx.y * 4 + kg; g < nkg; g += gridDim.y * 4) {
    double x[8];
    int t[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = g * 8 + j;
      t[j] = k < b.k ? balance<BAL>(b, kx, kexp, k) : 0;
      x[j] = (r < b.rows && k < b.k)
                 ? (double)X[b.kcont ? (int64_t)r * b.ld + k : r + (int64_t)k * b.ld]
                 : 0.0;
    }
    write_slices(x, s, t, W + (b.dst + g / 2) * BLK, r, g);
  }
}

// Exponents and slices in one pass, for products A A^T of up to ROW_K k: a thread
// keeps its row's entries (two groups of 8 k) in registers, the four threads of a
// row agree on its largest exponent.
constexpr int ROW_K = 64;
template <typename S>
__global__ void __launch_bounds__(256) k_f64_slice_rows(const SliceBlk* __restrict__ blks,
                                                        const S* __restrict__ Ab, int* exps,
                                                        unsigned char* W) {
  const SliceBlk b = blks[blockIdx.x];
  const S* X = Ab + b.src;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int r = warp * 8 + lane % 8, kg = lane / 8;
  double x[2][8];
  int m = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = (4 * h + kg) * 8 + j;
      x[h][j] = (r < b.rows && k < b.k)
                    ? (double)X[b.kcont ? (int64_t)r * b.ld + k : r + (int64_t)k * b.ld]
                    : 0.0;
      m = max(m, entry_exp(x[h][j], 0));
    }
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
  if (kg == 0) exps[(int64_t)blockIdx.x * BR + r] = m;
  const int s = row_exp(m);
  const int t[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int g = 4 * h + kg;
    if (g < (b.k + KC - 1) / KC * 2) write_slices(x[h], s, t, W + (b.dst + g / 2) * BLK, r, g);
  }
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, int bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(tc5::smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld4(uint32_t addr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr));
}

// (hi 2^32 + lo) 2^ex rounded to double (ties to even)
__device__ __forceinline__ double to_double(int64_t hi, int64_t lo, int ex) {
  // 128-bit two's complement of the sum: high and low 64 bits
  const uint64_t ul = (uint64_t)hi << 32;
  uint64_t l = ul + (uint64_t)lo;
  uint64_t h = (uint64_t)(hi >> 32) + (uint64_t)(lo >> 63) + (l < ul ? 1 : 0);
  const bool neg = (int64_t)h < 0;
  if (neg) {
    l = ~l + 1;
    h = ~h + (l == 0 ? 1 : 0);
  }
  if (h == 0 && l == 0) return 0.0;
  // leading bit to bit 63 of h, what falls off below kept as a sticky bit
  int lead = 0;
  if (h == 0) {
    h = l;
    l = 0;
    lead = 64;
  }
  const int z = __clzll((long long)h);
  lead += z;
  if (z) {
    h = (h << z) | (l >> (64 - z));
    l <<= z;
  }
  h |= l ? 1 : 0;
  uint64_t m = h >> 11;                       // 53 bits
  const uint32_t rem = (uint32_t)h & 0x7ff;
  m += (rem > 0x400 || (rem == 0x400 && (m & 1))) ? 1 : 0;
  const int e = 127 - lead + ex + 1023;       // biased exponent of bit 52 of m
  double v;
  if (e > 0 && e < 0x7fe) v = __longlong_as_double((long long)(((uint64_t)(e - 1) << 52) + m));
  else v = scalbn((double)(int64_t)m, e - 1023 - 52);
  return neg ? -v : v;
}

// NS: slices of each operand that are multiplied
template <int NS>
__global__ void __launch_bounds__(THREADS, 1)
    k_gemm_f64tc(const Tile* __restrict__ tiles, const GemmOp* __restrict__ ops,
                 const SliceBlk* __restrict__ blks, const int* __restrict__ exps,
                 const unsigned char* __restrict__ W, double* Cb, int* flags) {
  const Tile tl = tiles[blockIdx.x];
  const GemmOp o = ops[tl.op];
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[NST], done[NST], accf;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail, s_ea[TM], s_eb[TN];
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  if (tid < TM + TN) {   // the tile's row and column exponents
    const bool a = tid < TM;
    const int i = a ? tid : tid - TM;
    const int64_t at = (int64_t)(a ? tl.ablk : tl.bblk) * BR + i;
    const bool have = a ? tl.rb + i < o.m : tl.cb + i < o.n;
    (a ? s_ea : s_eb)[i] = have ? row_exp(exps[at]) : 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(
        tc5::smem_u32(&s_tmem)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc5::smem_u32(&full[s])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc5::smem_u32(&done[s])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(tc5::smem_u32(&accf)));
    asm volatile("fence.mbarrier_init.release.cluster;\n");
    asm volatile("fence.proxy.async.shared::cta;\n");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = s_tmem, sm0 = tc5::smem_u32(smem);
  int kbeg, kend;
  gemm_k_range(o, tl.rb, TM, tl.cb, TN, &kbeg, &kend);   // kbeg: a multiple of 64
  const int b0 = kbeg / KC, nc = (kend + KC - 1) / KC - b0;
  const bool two = tl.rb + BR < o.m;                     // rows in A's second block
  const unsigned char* A0 = W + (blks[tl.ablk].dst + b0) * BLK;
  const unsigned char* A1 = two ? W + (blks[tl.ablk + 1].dst + b0) * BLK : A0;
  const unsigned char* B0 = W + (blks[tl.bblk].dst + b0) * BLK;

  auto wait = [&](uint64_t* bar, uint32_t parity) {
    for (long long it = 0; it < WAIT_LIMIT; ++it)
      if (tc5::mbar_test(bar, parity)) return true;
    return false;
  };
  // warp 1: block c of both operands into its stage, one copy per lane.  A:
  // slice i's two halves of 64 rows next to each other; B: as stored.
  auto load = [&](int c) {
    const int s = c % NST;
    const uint32_t st = sm0 + s * STAGE;
    if (lane == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(
                       tc5::smem_u32(&full[s])),
                   "r"((two ? 3 : 2) * NS * SLICE)
                   : "memory");
    __syncwarp();
    const int64_t off = (int64_t)c * BLK;
    if (lane < 2 * NS) {
      if (two || lane % 2 == 0)
        bulk_copy(st + lane * SLICE, (lane % 2 ? A1 : A0) + off + (lane / 2) * SLICE, SLICE, &full[s]);
    } else if (lane == 2 * NS) {
      bulk_copy(st + 2 * BLK, B0 + off, NS * SLICE, &full[s]);
    }
  };
  int loaded = 0;               // warp 1: blocks loaded
  int issued = 0, seen = 0;     // thread 0: blocks multiplied, seen complete
  if (warp == 1)
    for (; loaded < min(NST - 1, nc); ++loaded) load(loaded);

  // this thread's entries of the tile: one row, a quarter of the columns; their sums and
  // C go through the stages' shared memory at the end
  const int cr = tl.rb + (warp % 4) * 32 + lane, cc = tl.cb + (warp / 4) * CW;
  int64_t* sum = reinterpret_cast<int64_t*>(smem) + tid;
  double* cst = reinterpret_cast<double*>(smem + sizeof(int64_t) * 2 * CW * THREADS) + tid;
  static_assert(sizeof(int64_t) * 2 * CW * THREADS + sizeof(double) * CW * THREADS <= NST * STAGE,
                "sums and C fit the stages");
  int64_t hi[CW], lo[CW];
#pragma unroll
  for (int j = 0; j < CW; ++j) hi[j] = lo[j] = 0;
  bool ok = true;
  const int ngroup = (nc + GROUP - 1) / GROUP;
  for (int g = 0; g < ngroup; ++g) {
    const int c1 = min(nc, (g + 1) * GROUP);
    if (tid == 0) {
      for (int c = g * GROUP; c < c1; ++c) {
        const int s = c % NST;
        if (!wait(&full[s], (c / NST) & 1)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        const uint32_t a = sm0 + s * STAGE, b = a + 2 * BLK;
        // slices j .. j + w - 1 of B lie one after the other, as do the
        // accumulators t = i + j .. they add to: one instruction of N = 64 w
        const uint64_t da = tc5::sdesc(a, 128, 256), db = tc5::sdesc(b, 128, 256);
        const uint32_t more = c > g * GROUP ? 1u : 0u;
#pragma unroll
        for (int i = 0; i < NS; ++i)
#pragma unroll
          for (int j = 0; i + j < NS; j += 4) {
            const int w = NS - i - j < 4 ? NS - i - j : 4;
            tc5::mma_bf16(tmem + (i + j) * TN, da + (2 * i * SLICE >> 4), db + (j * SLICE >> 4),
                          tc5::idesc_bf16(TM, w * TN), i > 0 ? 1u : more);
          }
        tc5::commit(&done[s]);
        ++issued;
      }
      if (ok) tc5::commit(&accf);
      else atomicExch(&s_fail, 1);
    } else if (warp == 1) {
      // three blocks ahead: the stage is free once the block before c is done
      for (int c = g * GROUP; c < c1 && loaded < nc; ++c) {
        const bool is_free = c == 0 || wait(&done[(c - 1) % NST], ((c - 1) / NST) & 1);
        if (!__all_sync(0xffffffffu, is_free)) {
          ok = false;
          atomicExch(&s_fail, 1);
          break;
        }
        load(loaded++);
      }
    }
    __syncwarp();   // the rest of warp 0 must not poll (and suspend it) while thread 0 issues
    if (ok) {
      ok = false;
      for (long long it = 0; it < WAIT_LIMIT && !*(volatile int*)&s_fail; ++it)
        if (tc5::mbar_test(&accf, g & 1)) {
          ok = true;
          break;
        }
    }
    // one verdict for the CTA: the loads from tensor memory are warp-collective
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    seen = issued;
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    if (g == ngroup - 1 && o.beta != 0.f) {
      // every copy and product is done: C arrives in the free stages while the
      // last accumulators are read back
#pragma unroll 4
      for (int j = 0; j < CW; ++j) {
        const bool in = cr < o.m && cc + j < o.n;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(
                         tc5::smem_u32(cst + j * THREADS)),
                     "l"(in ? Cb + o.C + cr + (int64_t)(cc + j) * o.ldc : Cb), "r"(in ? 8 : 0)
                     : "memory");
      }
    }
    const uint32_t base = tmem + ((uint32_t)((warp % 4) * 32) << 16) + (uint32_t)(warp / 4) * CW;
#pragma unroll
    for (int c0 = 0; c0 < CW; c0 += 4) {
      uint32_t d[NSL][4];
#pragma unroll
      for (int t = 0; t < NS; ++t) tmem_ld4(base + t * TN + c0, d[t]);
      asm volatile("tcgen05.wait::ld.sync.aligned;\n");
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        auto v = [&](int t) { return (int64_t)__float2int_rz(__uint_as_float(d[t][j])); };
        hi[c0 + j] += (v(0) << 24) + (v(1) << 16) + (v(2) << 8) + v(3);
        lo[c0 + j] += (v(4) << 24) + (v(5) << 16) + (v(6) << 8) + (NS == NSL ? v(NSL - 1) : 0);
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
  }
  if (!ok) {
    // drain, again bounded: copies that may still arrive, products still running
    if (warp == 1)
      for (int c = max(0, loaded - NST); c < loaded; ++c) wait(&full[c % NST], (c / NST) & 1);
    if (tid == 0) {
      for (int c = max(seen, issued - NST); c < issued; ++c) wait(&done[c % NST], (c / NST) & 1);
      atomicCAS(&flags[FLAG_TIMEOUT], -1, tl.op);
    }
  }
  if (ok) {
    // one short loop rounds the sums: unrolled over the registers it was 32
    // copies of the rounding, and fetching them took 30 us
#pragma unroll
    for (int j = 0; j < CW; ++j) {
      sum[(2 * j) * THREADS] = hi[j];
      sum[(2 * j + 1) * THREADS] = lo[j];
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    if (cr < o.m) {
      const int ea = s_ea[cr - tl.rb];
      double* C = Cb + o.C + cr + (int64_t)cc * o.ldc;
      const double al = (double)o.alpha;
      const int nj = min(CW, o.n - cc);
      const int* ebp = s_eb + (cc - tl.cb);
#pragma unroll 4
      for (int j = 0; j < nj; ++j) {
        const int eb = ebp[j];
        // 2^(sA - 63) 2^(sB - 63) 256^7, the biased exponents' offset 2 * 1023 taken out
        const double v = ea == NOT_FINITE || eb == NOT_FINITE
                             ? __longlong_as_double(0x7ff8000000000000ll)
                             : to_double(sum[(2 * j) * THREADS], sum[(2 * j + 1) * THREADS],
                                         ea + eb - 2 * 1023 - 126 + 56);
        C[(int64_t)j * o.ldc] = o.beta != 0.f ? fma(al, v, ngroup ? cst[j * THREADS] : C[(int64_t)j * o.ldc])
                                              : al * v;
      }
    }
  }
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

}  // namespace

// One 64 x 64 tile of the FMA form takes 1.2 us per k on its SM; the launches and one
// tile here take 28 to 34 us, whatever the k up to 100.
bool f64tc_worth(const GemmOp* h_ops, int nops) {
  for (int i = 0; i < nops; ++i)
    if (h_ops[i].k >= 24 && (int64_t)h_ops[i].m * h_ops[i].n >= 1024) return true;
  return false;
}

template <typename S>
void gemm_f64tc(const GemmOp* d_ops, const GemmOp* h_ops, int nops, const S* Abase, const S* Bbase,
                double* Cbase, int* d_flags, cudaStream_t st, const char* name, const int* d_kexp) {
  static const bool attr = [] {   // initialised once, also under concurrent factorizations
    HIF_CUDA_TRY(cudaFuncSetAttribute(k_gemm_f64tc<slices_used<S>()>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      NST * STAGE));
    return true;
  }();
  (void)attr;
  for (int f0 = 0; f0 < nops;) {
    // the products whose slices fit the work space together (at least one)
    std::vector<SliceBlk> blks;
    std::vector<Tile> tiles;
    int64_t nblk = 0, nkx = 0;
    double fl = 0;
    int f = f0, kmax = 0;
    bool all_same = true, balanced = false;
    for (; f < nops; ++f) {
      const GemmOp& o = h_ops[f];
      const int nk = ceil_div(o.k, KC);
      const bool same = Abase == Bbase && o.A == o.B && o.lda == o.ldb && o.transA != o.transB;
      const int na = ceil_div(o.m, BR), nb = ceil_div(o.n, BR);
      const int64_t need = (int64_t)(same ? std::max(na, nb) : na + nb) * nk;
      if (f > f0 && (size_t)(nblk + need) * BLK > WORK_LIMIT) break;
      const int kbal = same ? KB_NONE : o.kbal;
      all_same = all_same && same;
      balanced = balanced || kbal != KB_NONE;
      auto add = [&](int64_t src, int rows, int ld, bool kcont, bool isB) {
        const int first = (int)blks.size();
        for (int r0 = 0; r0 < rows; r0 += BR) {
          blks.push_back(SliceBlk{src + (kcont ? (int64_t)r0 * ld : r0), nblk, kbal == KB_MAX ? nkx : o.ks, ld,
                                  std::min(BR, rows - r0), o.k, kcont ? 1 : 0, isB ? 1 : 0, kbal});
          nblk += nk;
        }
        return first;
      };
      const int fa = add(o.A, same ? std::max(o.m, o.n) : o.m, o.lda, o.transA != 0, false);
      const int fb = same ? fa : add(o.B, o.n, o.ldb, o.transB == 0, true);
      if (kbal == KB_MAX) nkx += 2 * (int64_t)o.k;
      const int tm = ceil_div(o.m, TM), tn = ceil_div(o.n, TN);
      for (int t = 0; t < tm * tn; ++t) {
        const int q = gemm_tile(o, t, tm * tn);
        const int rb = (q % tm) * TM, cb = (q / tm) * TN;
        if (o.lower && cb >= rb + TM) continue;
        tiles.push_back(Tile{f, rb, cb, fa + rb / BR, fb + cb / BR});
      }
      kmax = std::max(kmax, o.k);
      fl += 2.0 * o.m * (double)o.n * o.k * (o.lower || o.kzero ? 0.5 : 1.0);
    }
    ProfScope ps(name, st, fl, 0.0);
    const size_t bb = sizeof(SliceBlk) * blks.size(), tb = sizeof(Tile) * tiles.size();
    DevBuf tab_b, work_b, exps_b;
    unsigned char* d_tab = tab_b.scratch<unsigned char>(bb + tb, st);
    unsigned char* W = work_b.scratch<unsigned char>((size_t)nblk * BLK, st);
    const size_t eb = sizeof(int) * (BR * blks.size() + (size_t)nkx);   // exps, then kx
    int* d_exps = exps_b.scratch<int>(eb / sizeof(int), st);
    int* d_kx = d_exps + BR * blks.size();
    std::vector<unsigned char> tab(bb + tb);
    std::copy_n(reinterpret_cast<const unsigned char*>(blks.data()), bb, tab.data());
    std::copy_n(reinterpret_cast<const unsigned char*>(tiles.data()), tb, tab.data() + bb);
    HIF_CUDA_TRY(cudaMemcpyAsync(d_tab, tab.data(), bb + tb, cudaMemcpyHostToDevice, st));
    const SliceBlk* d_blks = reinterpret_cast<const SliceBlk*>(d_tab);
    const Tile* d_tiles = reinterpret_cast<const Tile*>(d_tab + bb);
    const int gy = std::max(1, std::min({ceil_div(kmax, 64), 64, ceil_div(4096, (int64_t)blks.size())}));
    const bool rows = all_same && kmax <= ROW_K;
    if (rows) {
      k_f64_slice_rows<S><<<(unsigned)blks.size(), 256, 0, st>>>(d_blks, Abase, d_exps, W);
      HIF_CHECK_LAUNCH();
    } else {
      const dim3 grid((unsigned)blks.size(), gy);
      HIF_CUDA_TRY(cudaMemsetAsync(d_exps, 0, eb, st));
      if (nkx) {
        k_f64_kmax<S><<<grid, 256, 0, st>>>(d_blks, Abase, Bbase, d_kx);
        HIF_CHECK_LAUNCH();
      }
      (balanced ? k_f64_exps<S, true> : k_f64_exps<S, false>)<<<grid, 256, 0, st>>>(
          d_blks, Abase, Bbase, d_kx, d_kexp, d_exps);
      HIF_CHECK_LAUNCH();
      (balanced ? k_f64_slice<S, true> : k_f64_slice<S, false>)<<<grid, 256, 0, st>>>(
          d_blks, Abase, Bbase, d_kx, d_kexp, d_exps, W);
      HIF_CHECK_LAUNCH();
    }
    k_gemm_f64tc<slices_used<S>()><<<(unsigned)tiles.size(), THREADS, NST * STAGE, st>>>(
        d_tiles, d_ops, d_blks, d_exps, W, Cbase, d_flags);
    HIF_CHECK_LAUNCH();
    f0 = f;
  }
}

template void gemm_f64tc<double>(const GemmOp*, const GemmOp*, int, const double*, const double*,
                                 double*, int*, cudaStream_t, const char*, const int*);
template void gemm_f64tc<float>(const GemmOp*, const GemmOp*, int, const float*, const float*,
                                double*, int*, cudaStream_t, const char*, const int*);

}  // namespace hif
