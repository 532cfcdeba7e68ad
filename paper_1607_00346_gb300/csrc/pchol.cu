// Interpolative decomposition of FP32 faces with many coupled rows, from their
// Gram matrix in FP64.
//
// The ID of A_RF (§2.3) depends on A_RF only through the norms of combinations of
// its columns, so the pivots and the R factor of its column-pivoted QR are those
// of the pivoted Cholesky factorization G = A_RF^T A_RF = P R^T R P^T: each step
// takes the column with the largest remaining diagonal entry, |R_ii|^2, and
// subtracts the outer product of its row of R.  Squaring the matrix squares its
// condition number, so G needs twice the digits: it is formed from the FP32 entries,
// cut 55 bits below the largest of their column, with sums off by less than 2^-50 of the
// two columns' largest entries per row (f64tc.cu: seven slices), and factored in FP64,
// which leaves R_ii an error of 1e-8 |R_11|, where Householder QR in FP32 leaves 6e-8.
// Pivots below that are noise whose rows of R need not be bounded by them (QR's are), so
// fronts with a smaller eps than GRAM_EPS stay with the row reduction and QR: FP32 at
// eps 1e-12, a = 10^U(-2,2), the Gram form lost 250 times the solve error at 48^3 and
// failed at 64^3; at 1e-10 it kept 3% fewer skeletons; at 1e-7 and above it keeps the
// same ones.
//
// What it replaces is bound by chains: the unpivoted QR of the tall A_RF column by
// column (two barriers and a pass over a 32-column panel each), then pivoted QR of
// R, whose every step reads the trailing matrix once.  Here the tall matrix is
// read once, by tensor-core products, and a pivot step reads one column of G: 64
// steps per launch in k_pchol (a cluster per front, one column per thread), then
// one product per front updates G.  128^3, FP32, eps 1e-6: row reduction and ID of
// the three upper levels' faces 300 ms, here 89 ms (56 + 15 the products, 18 the
// steps; 48 steps per launch: 19.5 + 21 instead of 15 + 26 before the comparisons
// and reciprocal roots left the FP64 unit, 32 steps: 27.5 + 18).
#include <algorithm>
#include <climits>
#include <vector>

#include <cooperative_groups.h>

#include "common.cuh"
#include "dense.cuh"
#include "front.cuh"
#include "pchol.cuh"

namespace hif {

namespace cg = cooperative_groups;

namespace {

constexpr double GRAM_EPS = 1e-7;  // the least eps whose pivots G resolves
constexpr int PC_STEPS = 64;       // pivots per launch
// A CTA of 128 columns keeps 64 KB of the block's rows, so that three share an SM and
// one's barriers overlap the others' sums; 256 columns (one per SM, 128 KB) for fronts
// of more than 1024 columns, which 8 CTAs of 128 do not hold.  128^3, eps 1e-6: 18.4
// against 19.7 ms with 256 throughout; eps 1e-3: 7.2 against 8.9; 96^3: 7.4 and 7.3.
constexpr int PC_NARROW = 128, PC_NARROW_CS = 8;
constexpr int PC_WIDE = 256, PC_WIDE_CS = 16;
constexpr size_t pc_smem(int threads) { return sizeof(double) * PC_STEPS * threads; }

struct PcDesc {
  int64_t G;       // n x n (lower triangle), in the Gram arena
  int64_t L;       // n x PC_STEPS, in the block arena
  int64_t R;       // offset in the R arena (leading dimension n)
  int64_t col;     // first entry of its columns' state
  int64_t perm;    // offset of its permutation
  int n, front;    // front: index in the SkelDesc array
};

struct PcState {
  double d1;       // the first pivot's diagonal, |R_11|^2
  int k, done;     // pivots so far; no further ones
};

__global__ void k_pchol_init(const PcDesc* __restrict__ ds, const double* __restrict__ G,
                             double* diag, int* step, PcState* stt) {
  const PcDesc d = ds[blockIdx.x];
  for (int c = threadIdx.x; c < d.n; c += blockDim.x) {
    diag[d.col + c] = G[d.G + c + (int64_t)c * d.n];
    step[d.col + c] = -1;
  }
  if (threadIdx.x == 0) stt[blockIdx.x] = PcState{0.0, 0, 0};
}

// The larger of two diagonals, the lower column on ties.  Diagonals are compared as
// integers: positive doubles are ordered like their bits and above all negative ones,
// and a comparison on the FP64 unit (16 clocks a warp) costs as much as an FMA.
__device__ __forceinline__ bool larger(long long& bd, int& bc, long long od, int oc) {
  const bool take = od > bd || (od == bd && oc < bc);
  if (take) {
    bd = od;
    bc = oc;
  }
  return take;
}

// PC_STEPS pivots of each listed front: column c belongs to thread c % PC_THREADS of
// CTA c / PC_THREADS of its cluster, which keeps its remaining diagonal in a register and its
// entries of the block's rows of R in shared memory.  Per step every CTA proposes
// its largest diagonal, with that column's entries of the block so far, to all
// CTAs of the cluster; after one cluster barrier all pick the same winner
// (largest, lowest column on ties) and each thread forms its entry of the new row,
// (G_cp - sum of the block's products) / R_pp.  What bounds it is the FP64 unit (2 per
// clock and SM): comparisons are on integers, and 1 / R_pp comes with the proposal
// (128^3: 26.0 -> 18.4 ms, 96^3: 9.6 -> 7.4 ms, against both in every thread).
template <int PC_THREADS, int PC_MAX_CS>
__global__ void __launch_bounds__(PC_THREADS) k_pchol(const PcDesc* __restrict__ ds,
                                                     const int* __restrict__ list,
                                                     const double* __restrict__ Gar, double* Lar,
                                                     float* Rar, double* diag, int* step,
                                                     PcState* stt, double eps2) {
  constexpr int PC_WARPS = PC_THREADS / 32;
  cg::cluster_group cl = cg::this_cluster();
  const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int f = list[blockIdx.x / CS];
  const PcDesc d = ds[f];
  const int n = d.n, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int c = rank * PC_THREADS + tid;
  const bool in = c < n;
  extern __shared__ __align__(16) unsigned char psm[];
  double(*Lb)[PC_THREADS] = reinterpret_cast<double(*)[PC_THREADS]>(psm);
  __shared__ double s_binv[2][PC_MAX_CS], s_row[2][PC_MAX_CS][PC_STEPS];
  __shared__ long long s_bd[2][PC_MAX_CS];
  __shared__ int s_bc[2][PC_MAX_CS];
  __shared__ long long w_d[PC_WARPS];
  __shared__ int w_c[PC_WARPS];
  const double* G = Gar + d.G;
  double dc = in ? diag[d.col + c] : 0.0;
  int tk = in ? step[d.col + c] : 0;
  const PcState s0 = stt[f];
  double d1 = s0.d1, least = eps2 * d1;
  bool done = false;
  int j = 0;
  cl.sync();   // every CTA of the cluster runs before the first push
  for (; j < PC_STEPS; ++j) {
    const int par = j & 1;
    long long bd = tk < 0 ? __double_as_longlong(dc) : LLONG_MIN;
    int bc = c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) larger(bd, bc, __shfl_xor_sync(0xffffffffu, bd, o),
                                            __shfl_xor_sync(0xffffffffu, bc, o));
    if (lane == 0) {
      w_d[warp] = bd;
      w_c[warp] = bc;
    }
    __syncthreads();   // also: every thread's entry of the last row is in Lb
    if (warp == 0) {
      bd = w_d[lane % PC_WARPS];
      bc = w_c[lane % PC_WARPS];
#pragma unroll
      for (int o = PC_WARPS / 2; o > 0; o >>= 1) larger(bd, bc, __shfl_xor_sync(0xffffffffu, bd, o),
                                                        __shfl_xor_sync(0xffffffffu, bc, o));
      const double binv = rsqrt(__longlong_as_double(bd));
      for (int q = 0; q < CS; ++q) {
        for (int t = lane; t < j; t += 32)
          *cl.map_shared_rank(&s_row[par][rank][t], q) = Lb[t][bc - rank * PC_THREADS];
        if (lane == 0) {
          *cl.map_shared_rank(&s_bd[par][rank], q) = bd;
          *cl.map_shared_rank(&s_binv[par][rank], q) = binv;
          *cl.map_shared_rank(&s_bc[par][rank], q) = bc;
        }
      }
    }
    cl.sync();
    long long mk = s_bd[par][0];
    int mc = s_bc[par][0], mr = 0;
    for (int q = 1; q < CS; ++q)
      if (larger(mk, mc, s_bd[par][q], s_bc[par][q])) mr = q;
    const double md = __longlong_as_double(mk);
    if (s0.k + j == 0) {
      d1 = md;
      least = eps2 * d1;
    }
    if (mk <= 0 || mk <= __double_as_longlong(least) || mk >= 0x7ff0000000000000ll) {
      done = true;
      break;
    }
    double l = 0.0;
    if (tk < 0) {
      const double inv = s_binv[par][mr];
      const double g = c >= mc ? G[c + (int64_t)mc * n] : G[mc + (int64_t)c * n];
      const double* row = s_row[par][mr];
      double t0 = g, t1 = 0.0, t2 = 0.0, t3 = 0.0;
      int q = 0;
      for (; q + 4 <= j; q += 4) {
        t0 = fma(-Lb[q][tid], row[q], t0);
        t1 = fma(-Lb[q + 1][tid], row[q + 1], t1);
        t2 = fma(-Lb[q + 2][tid], row[q + 2], t2);
        t3 = fma(-Lb[q + 3][tid], row[q + 3], t3);
      }
      for (; q < j; ++q) t0 = fma(-Lb[q][tid], row[q], t0);
      l = ((t0 + t1) + (t2 + t3)) * inv;
      if (c == mc) {
        l = md * inv;
        tk = s0.k + j;
      } else {
        dc = fma(-l, l, dc);
      }
    }
    Lb[j][tid] = l;
  }
  cl.sync();   // no CTA leaves while another may still read its proposal
  if (in) {
    for (int q = 0; q < PC_STEPS; ++q) Lar[d.L + c + (int64_t)q * n] = q < j ? Lb[q][tid] : 0.0;
    float* R = Rar + d.R + s0.k + (int64_t)c * n;
    for (int q = 0; q < j; ++q) R[q] = (float)Lb[q][tid];
    diag[d.col + c] = dc;
    step[d.col + c] = tk;
  }
  if (rank == 0 && tid == 0) stt[f] = PcState{d1, s0.k + j, done || s0.k + j == n ? 1 : 0};
}

// the pivots in order, then the other columns in increasing order
constexpr int PERM_THREADS = 256;
__global__ void __launch_bounds__(PERM_THREADS) k_pchol_perm(const PcDesc* __restrict__ ds,
                                                          const int* __restrict__ step,
                                                          const PcState* __restrict__ stt,
                                                          int32_t* perm, SkelDesc* fr) {
  const PcDesc d = ds[blockIdx.x];
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  int32_t* pv = perm + d.perm;
  __shared__ int s_cnt[PERM_THREADS / 32];
  int base = stt[blockIdx.x].k;
  if (tid == 0) fr[d.front].k = base;
  for (int c0 = 0; c0 < d.n; c0 += PERM_THREADS) {
    const int c = c0 + tid;
    const int t = c < d.n ? step[d.col + c] : 0;
    const bool left = c < d.n && t < 0;
    const unsigned m = __ballot_sync(0xffffffffu, left);
    if (lane == 0) s_cnt[warp] = __popc(m);
    __syncthreads();
    int before = base, all = 0;
    for (int w = 0; w < PERM_THREADS / 32; ++w) {
      before += w < warp ? s_cnt[w] : 0;
      all += s_cnt[w];
    }
    if (left) pv[before + __popc(m & ((1u << lane) - 1u))] = c;
    else if (c < d.n) pv[t] = c;
    base += all;
    __syncthreads();
  }
}

// Cluster sizes of k_pchol<THREADS, MAX_CS> that can be resident (index: size)
template <int THREADS, int MAX_CS>
const std::vector<int>& pchol_placeable() {
  static const std::vector<int> placeable = [] {
    auto* k = k_pchol<THREADS, MAX_CS>;
    HIF_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    HIF_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)pc_smem(THREADS)));
    std::vector<int> ok(MAX_CS + 1, 0);
    for (int s = 1; s <= MAX_CS; ++s) {
      cudaLaunchConfig_t q = {};
      q.gridDim = dim3((unsigned)s);
      q.blockDim = dim3(THREADS);
      q.dynamicSmemBytes = pc_smem(THREADS);
      cudaLaunchAttribute qa[1];
      qa[0].id = cudaLaunchAttributeClusterDimension;
      qa[0].val.clusterDim.x = s;
      qa[0].val.clusterDim.y = 1;
      qa[0].val.clusterDim.z = 1;
      q.attrs = qa;
      q.numAttrs = 1;
      int ncl = 0;
      ok[s] = cudaOccupancyMaxActiveClusters(&ncl, k, &q) == cudaSuccess && ncl > 0;
      cudaGetLastError();
    }
    return ok;
  }();
  return placeable;
}

// CTAs of 128 columns for a batch whose largest front has n columns
bool pchol_narrow(int n) {
  const int cs = ceil_div(n, PC_NARROW);
  return cs <= PC_NARROW_CS && pchol_placeable<PC_NARROW, PC_NARROW_CS>()[cs] != 0;
}

}  // namespace

bool gram_id_fits(int nFmax, double eps) {
  if (eps < GRAM_EPS) return false;
  if (pchol_narrow(nFmax)) return true;
  const int cs = ceil_div(nFmax, PC_WIDE);
  return cs <= PC_WIDE_CS && pchol_placeable<PC_WIDE, PC_WIDE_CS>()[cs] != 0;
}

void gram_id(SkelDesc* d_f, const SkelDesc* h_f, int nf, const float* Garena, float* Rout,
             int32_t* perm, double eps, int* d_flags, cudaStream_t st) {
  if (nf == 0) return;
  std::vector<PcDesc> ds(nf);
  std::vector<GemmOp> ops(nf);
  int64_t gt = 0, lt = 0, ct = 0;
  int nmax = 1;
  for (int f = 0; f < nf; ++f) {
    const SkelDesc& s = h_f[f];
    ds[f] = PcDesc{gt, lt, s.idoff, ct, s.perm, s.nF, f};
    ops[f] = GemmOp{s.G + s.nF, s.G + s.nF, gt, s.nF, s.nF, s.nR, s.nF + s.nR, s.nF + s.nR, s.nF, 1, 0,
                    1.f, 0.f, 1, 0};
    gt += (int64_t)s.nF * s.nF;
    lt += (int64_t)s.nF * PC_STEPS;
    ct += s.nF;
    nmax = std::max(nmax, s.nF);
  }
  const bool narrow = pchol_narrow(nmax);
  const int threads = narrow ? PC_NARROW : PC_WIDE, CS = ceil_div(nmax, threads);
  DevBuf G, L, diag, step, stt, dds, dop, lst;
  G.scratch<double>(gt, st);
  L.scratch<double>(lt, st);
  diag.scratch<double>(ct, st);
  step.scratch<int>(ct, st);
  stt.scratch<PcState>(nf, st);
  dds.scratch<PcDesc>(nf, st);
  dop.scratch<GemmOp>(nf, st);
  lst.scratch<int>(nf, st);
  HIF_CUDA_TRY(cudaMemcpyAsync(dds.as<void>(), ds.data(), sizeof(PcDesc) * nf, cudaMemcpyHostToDevice, st));
  HIF_CUDA_TRY(cudaMemcpyAsync(dop.as<void>(), ops.data(), sizeof(GemmOp) * nf, cudaMemcpyHostToDevice, st));
  gemm_f64tc<float>(dop.as<GemmOp>(), ops.data(), nf, Garena, Garena, G.as<double>(), d_flags, st,
                    "id_gram_f64tc");
  {
    ProfScope ps("id_pchol", st);
    k_pchol_init<<<nf, 256, 0, st>>>(dds.as<PcDesc>(), G.as<double>(), diag.as<double>(),
                                    step.as<int>(), stt.as<PcState>());
    HIF_CHECK_LAUNCH();
  }
  std::vector<int> act(nf);
  for (int f = 0; f < nf; ++f) act[f] = f;
  std::vector<PcState> h(nf);
  while (!act.empty()) {
    HIF_CUDA_TRY(cudaMemcpyAsync(lst.as<void>(), act.data(), sizeof(int) * act.size(), cudaMemcpyHostToDevice, st));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(act.size() * CS));
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = pc_smem(threads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    {
      ProfScope ps("id_pchol", st);
      HIF_CUDA_TRY(cudaLaunchKernelEx(&cfg, narrow ? k_pchol<PC_NARROW, PC_NARROW_CS> : k_pchol<PC_WIDE, PC_WIDE_CS>,
                                      (const PcDesc*)dds.as<PcDesc>(),
                                      (const int*)lst.as<int>(), (const double*)G.as<double>(),
                                      L.as<double>(), Rout, diag.as<double>(), step.as<int>(),
                                      stt.as<PcState>(), eps * eps));
      HIF_CHECK_LAUNCH();
    }
    HIF_CUDA_TRY(cudaMemcpyAsync(h.data(), stt.as<void>(), sizeof(PcState) * nf, cudaMemcpyDeviceToHost, st));
    HIF_CUDA_TRY(cudaStreamSynchronize(st));
    std::vector<int> next;
    for (int f : act)
      if (!h[f].done) next.push_back(f);
    act.swap(next);
    if (act.empty()) break;
    // G -= L L^T of the fronts that go on
    std::vector<GemmOp> up(act.size());
    for (size_t i = 0; i < act.size(); ++i) {
      const PcDesc& d = ds[act[i]];
      up[i] = GemmOp{d.L, d.L, d.G, d.n, d.n, PC_STEPS, d.n, d.n, d.n, 0, 1, -1.f, 1.f, 1, 0};
    }
    HIF_CUDA_TRY(cudaMemcpyAsync(dop.as<void>(), up.data(), sizeof(GemmOp) * up.size(), cudaMemcpyHostToDevice, st));
    gemm_f64tc<double>(dop.as<GemmOp>(), up.data(), (int)up.size(), L.as<double>(), L.as<double>(),
                       G.as<double>(), d_flags, st, "id_pchol_update_f64tc");
  }
  k_pchol_perm<<<nf, PERM_THREADS, 0, st>>>(dds.as<PcDesc>(), step.as<int>(), stt.as<PcState>(), perm, d_f);
  HIF_CHECK_LAUNCH();
}

}  // namespace hif
