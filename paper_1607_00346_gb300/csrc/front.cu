// Moving matrix entries between fronts: stencil coefficients (§2.4), level-0
// frontal matrices, extend-add of the children into a parent cell (the merge
// of §3.2, done in device memory), the gather of A_{[F;R],F} for a face or
// edge (§2.3) and the write-back of B_{F^F^}.
//
// Frontal matrices are symmetric; only their lower triangle is read or written
// (entry (a,b) lives at K[max(a,b) + min(a,b)*n]).
#include <algorithm>

#include "front.cuh"

namespace hif {

namespace {

constexpr int MAX_GRID_Y = 65535;

__device__ __forceinline__ double harmonic(double p, double q) { return 2.0 * p * q / (p + q); }

// Dirichlet: h = 1/(n+1), a neighbour outside the grid adds its coupling
// (a_j) to the diagonal only.  Periodic: h = 1/n, the last plane couples to
// the first, and b must be positive (otherwise the constant is a null vector).
__global__ void k_stencil(const double* __restrict__ a, const double* __restrict__ b,
                          double b_const, int n, int periodic, double* cpl, double* diag,
                          int* bad) {
  const int64_t N = (int64_t)n * n * n;
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= N) return;
  const int x[3] = {(int)(j % n), (int)((j / n) % n), (int)(j / ((int64_t)n * n))};
  const int64_t stride[3] = {1, n, (int64_t)n * n};
  const double h = periodic ? 1.0 / n : 1.0 / (n + 1);
  const double ih2 = 1.0 / (h * h);
  const double aj = a[j];
  const double bj = b ? b[j] : b_const;
  if (!(aj > 0.0) || !isfinite(aj) || !(bj >= 0.0) || !isfinite(bj) || (periodic && !(bj > 0.0)))
    atomicExch(bad, 1);
  double s = 0.0;
  for (int d = 0; d < 3; ++d) {
    double cm, cp;
    if (periodic) {
      const int64_t jm = x[d] > 0 ? j - stride[d] : j + (int64_t)(n - 1) * stride[d];
      const int64_t jp = x[d] + 1 < n ? j + stride[d] : j - (int64_t)(n - 1) * stride[d];
      cm = harmonic(a[jm], aj);
      cp = harmonic(aj, a[jp]);
      cpl[d * N + j] = cp * ih2;
    } else {
      cm = x[d] > 0 ? harmonic(a[j - stride[d]], aj) : aj;
      cp = x[d] + 1 < n ? harmonic(aj, a[j + stride[d]]) : aj;
      cpl[d * N + j] = x[d] + 1 < n ? cp * ih2 : 0.0;
    }
    s += cm + cp;
  }
  diag[j] = s * ih2 + bj;
}

// Positive doubles are ordered like their bits.
__global__ void __launch_bounds__(256) k_value_range(const double* __restrict__ a, int64_t cnt,
                                                     unsigned long long* range) {
  unsigned long long lo = ~0ull, hi = 0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * 256) {
    const unsigned long long v = (unsigned long long)__double_as_longlong(a[i]);
    lo = min(lo, v);
    hi = max(hi, v);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (threadIdx.x % 32 == 0) {
    atomicMin(&range[0], lo);
    atomicMax(&range[1], hi);
  }
}

// The cell (coordinate along one dimension) that owns point x at cell side
// s: a separator plane belongs to the cell below it (wrapping to the last
// cell on the periodic grid, where plane 0 is a separator too).
__device__ __forceinline__ int lowcell(int x, int s, int C, int periodic) {
  if (periodic) return x % s == 0 ? (x / s + C - 1) % C : x / s;
  return (x != 0 && x % s == 0) ? x / s - 1 : x / s;
}

// The cell's closure is the box [s c, s (c+1)] per dimension (clipped to the
// grid with a Dirichlet boundary, wrapping to plane 0 on the periodic grid);
// points are addressed by their offset from the box's low corner.
template <typename T>
__global__ void k_assemble0(const CellDesc* __restrict__ cells, const int32_t* __restrict__ lists,
                            int n, int s, int periodic, const double* __restrict__ cpl,
                            const double* __restrict__ diag, T* Kar) {
  extern __shared__ int boxmap[];
  const CellDesc cd = cells[blockIdx.x];
  const int C = n / s;
  const int c[3] = {(int)(blockIdx.x % C), (int)((blockIdx.x / C) % C), (int)(blockIdx.x / (C * C))};
  int lo[3], B[3];
  for (int d = 0; d < 3; ++d) {
    lo[d] = s * c[d];
    B[d] = periodic ? s + 1 : min(s * (c[d] + 1), n - 1) - lo[d] + 1;
  }
  const int32_t* lst = lists + cd.list;
  const int64_t N = (int64_t)n * n * n;
  for (int a = threadIdx.x; a < cd.n; a += blockDim.x) {
    const int g = lst[a];
    const int x[3] = {g % n, (g / n) % n, g / (n * n)};
    int xl[3];
    for (int d = 0; d < 3; ++d) xl[d] = (x[d] - lo[d] + n) % n;
    boxmap[xl[0] + B[0] * (xl[1] + B[1] * xl[2])] = a;
  }
  __syncthreads();
  T* K = Kar + cd.K;
  const int nc = cd.n;
  for (int a = threadIdx.x; a < nc; a += blockDim.x) {
    const int g = lst[a];
    const int x[3] = {g % n, (g / n) % n, g / (n * n)};
    int xl[3];
    for (int d = 0; d < 3; ++d) xl[d] = (x[d] - lo[d] + n) % n;
    bool own = true;
    for (int d = 0; d < 3; ++d) own = own && lowcell(x[d], s, C, periodic) == c[d];
    if (own) K[(int64_t)a + (int64_t)a * nc] = (T)diag[g];
    for (int d = 0; d < 3; ++d) {
      // the coupling of x with its +e_d neighbour, if the box holds both
      if (xl[d] + 1 >= B[d]) continue;
      bool ownp = x[d] / s == c[d];
      for (int e = 0; e < 3; ++e)
        if (e != d) ownp = ownp && lowcell(x[e], s, C, periodic) == c[e];
      if (!ownp) continue;
      int y[3] = {xl[0], xl[1], xl[2]};
      y[d] += 1;
      const int b = boxmap[y[0] + B[0] * (y[1] + B[1] * y[2])];
      const int hi_ = max(a, b), lo_ = min(a, b);
      K[(int64_t)hi_ + (int64_t)lo_ * nc] = (T)(-cpl[d * N + g]);
    }
  }
}

__device__ __forceinline__ void tri_index(int t, int& ti, int& tj) {
  int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (i * (i + 1) / 2 > t) --i;
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  ti = i;
  tj = t - i * (i + 1) / 2;
}

template <typename T>
__global__ void __launch_bounds__(256) k_merge(const MergeDesc* __restrict__ par,
                                               const CellDesc* __restrict__ child,
                                               const int32_t* __restrict__ maps,
                                               const T* __restrict__ Kc, T* Kp) {
  const MergeDesc pd = par[blockIdx.y];
  const int n = pd.n;
  const int nt = (n + 63) / 64;
  if ((int)blockIdx.x >= nt * (nt + 1) / 2) return;
  int ti, tj;
  tri_index(blockIdx.x, ti, tj);
  __shared__ int rmap[8][64];
  __shared__ int cmap[8][64];
  __shared__ int64_t cK[8];
  __shared__ int cn[8], cp[8];
  const int32_t* mp = maps + pd.map;
  for (int e = threadIdx.x; e < 8 * 64; e += 256) {
    const int q = e / 64, i = e % 64;
    const int a = ti * 64 + i, b = tj * 64 + i;
    const bool has = pd.child[q] >= 0;
    rmap[q][i] = (has && a < n) ? mp[(int64_t)q * n + a] : -1;
    cmap[q][i] = (has && b < n) ? mp[(int64_t)q * n + b] : -1;
  }
  if (threadIdx.x < 8) {
    const int ch = pd.child[threadIdx.x];
    if (ch >= 0) {
      const CellDesc cd = child[ch];
      cK[threadIdx.x] = cd.K;
      cn[threadIdx.x] = cd.n;
      cp[threadIdx.x] = cd.p;
    } else {
      cK[threadIdx.x] = 0;
      cn[threadIdx.x] = 0;
      cp[threadIdx.x] = 0;
    }
  }
  __syncthreads();
  // the children that hold row i / column j of the tile (bit q): an entry
  // visits only the children that hold both, in increasing q as before
  __shared__ unsigned s_rm[64], s_cm[64];
  if (threadIdx.x < 64) {
    unsigned r = 0u, c = 0u;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      r |= (rmap[q][threadIdx.x] >= 0 ? 1u : 0u) << q;
      c |= (cmap[q][threadIdx.x] >= 0 ? 1u : 0u) << q;
    }
    s_rm[threadIdx.x] = r;
    s_cm[threadIdx.x] = c;
  }
  __syncthreads();
  T* K = Kp + pd.K;
  for (int e = threadIdx.x; e < 64 * 64; e += 256) {
    const int i = e % 64, j = e / 64;
    const int a = ti * 64 + i, b = tj * 64 + j;
    if (a >= n || b >= n || a < b) continue;
    T sum = T(0);
    for (unsigned msk = s_rm[i] & s_cm[j]; msk != 0u; msk &= msk - 1u) {
      const int q = __ffs(msk) - 1;
      const int x = rmap[q][i], y = cmap[q][j];
      const int hi_ = max(x, y), lo_ = min(x, y);
      const int64_t ncq = cn[q], pq = cp[q];
      sum += Kc[cK[q] + (pq + hi_) + (pq + lo_) * ncq];
    }
    K[(int64_t)a + (int64_t)b * n] = sum;
  }
}

// One CTA per 32 x 32 tile of a front's gather block.  The cells' frontal
// matrices hold only their lower triangles, so an entry (x, y) with x < y is
// read as (y, x): the tile is accumulated in shared memory in two passes per
// cell, lanes over the tile's rows for the entries read down a column
// (x >= y) and lanes over its columns for the transposed ones (x < y), so
// both read consecutive addresses; the cells are added in order.  The kernel is
// bound by instructions, not by HBM, and most rows lie in one cell and on one
// side of the tile's columns: a pass that can hold no entry (from the least and
// largest positions of the tile's rows and columns) is left out.  128^3 FP32,
// 12 launches: 25.0 ms with every pass, 19.1 ms.
constexpr int GT = 32;   // gather tile

template <typename T>
__global__ void __launch_bounds__(256) k_skel_gather(const SkelDesc* __restrict__ fr, int ncp,
                                                     const int32_t* __restrict__ rowPos,
                                                     const CellDesc* __restrict__ cells,
                                                     const T* __restrict__ Kar, T* Gar) {
  const SkelDesc f = fr[blockIdx.y];
  const int rows = f.nF + f.nR, cols = f.nF;
  const int tr = (rows + GT - 1) / GT, tc = (cols + GT - 1) / GT;
  if ((int)blockIdx.x >= tr * tc) return;
  const int r0 = (int)(blockIdx.x % tr) * GT, c0 = (int)(blockIdx.x / tr) * GT;
  __shared__ T tile[GT][GT + 1];   // tile[c][r]
  __shared__ int xr[4][GT], yc[4][GT];
  __shared__ int64_t cK[4];
  __shared__ int cn[4], cp[4], pass[4];   // pass: bit 0 down a column, bit 1 transposed
  const int tx = threadIdx.x % GT, ty = threadIdx.x / GT;   // ty < 8
  const int32_t* rp = rowPos + f.rows;
  if (threadIdx.x < ncp) {
    const CellDesc cd = cells[f.cell[threadIdx.x]];
    cK[threadIdx.x] = cd.K;
    cn[threadIdx.x] = cd.n;
    cp[threadIdx.x] = cd.p;
  }
  if (ty < ncp) {
    const int x = r0 + tx < rows ? rp[(int64_t)(r0 + tx) * ncp + ty] : -1;
    const int y = c0 + tx < cols ? rp[(int64_t)(c0 + tx) * ncp + ty] : -1;
    xr[ty][tx] = x;
    yc[ty][tx] = y;
    const int xhi = __reduce_max_sync(0xffffffffu, x), yhi = __reduce_max_sync(0xffffffffu, y);
    const unsigned xlo = __reduce_min_sync(0xffffffffu, (unsigned)x);   // absent: the largest
    const unsigned ylo = __reduce_min_sync(0xffffffffu, (unsigned)y);
    if (tx == 0)
      pass[ty] = xhi < 0 || yhi < 0 ? 0 : ((unsigned)xhi >= ylo ? 1 : 0) | (xlo < (unsigned)yhi ? 2 : 0);
  }
  for (int q = ty; q < GT; q += 8) tile[q][tx] = T(0);
  __syncthreads();
  for (int i = 0; i < ncp; ++i) {
    const T* K = Kar + cK[i];
    const int64_t nc = cn[i], p = cp[i];
    if (pass[i] & 1) {
#pragma unroll
      for (int q = ty; q < GT; q += 8) {   // lanes over rows: (x, y) with x >= y
        const int x = xr[i][tx], y = yc[i][q];
        if (x >= 0 && y >= 0 && x >= y) tile[q][tx] += K[(p + x) + (p + y) * nc];
      }
      __syncthreads();
    }
    if (pass[i] & 2) {
#pragma unroll
      for (int q = ty; q < GT; q += 8) {   // lanes over columns: (x, y) with x < y, read as (y, x)
        const int x = xr[i][q], y = yc[i][tx];
        if (x >= 0 && y >= 0 && x < y) tile[tx][q] += K[(p + y) + (p + x) * nc];
      }
      __syncthreads();
    }
  }
  for (int q = ty; q < GT; q += 8)
    if (r0 + tx < rows && c0 + q < cols) Gar[f.G + (r0 + tx) + (int64_t)(c0 + q) * rows] = tile[q][tx];
}

template <typename T>
__global__ void __launch_bounds__(256) k_skel_permute(const SkelDesc* __restrict__ fr,
                                                      const int32_t* __restrict__ perm,
                                                      const T* __restrict__ Gar, T* Zar) {
  const SkelDesc f = fr[blockIdx.y];
  const int nF = f.nF;
  const int64_t tot = (int64_t)nF * nF;
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= tot) return;
  const int r = (int)(e % nF), c = (int)(e / nF);
  const int p = nF - f.k;
  const int32_t* pm = perm + f.perm;
  const int orr = r < p ? pm[f.k + r] : pm[r - p];
  const int occ = c < p ? pm[f.k + c] : pm[c - p];
  const int ld = nF + f.nR;
  Zar[f.Z + e] = Gar[f.G + orr + (int64_t)occ * ld];
}

template <typename T>
__global__ void __launch_bounds__(256) k_skel_writeback(const SkelDesc* __restrict__ fr, int ncp,
                                                        const int32_t* __restrict__ rowPos,
                                                        const int32_t* __restrict__ perm,
                                                        const CellDesc* __restrict__ cells,
                                                        const T* __restrict__ Zar, T* Kar) {
  const SkelDesc f = fr[blockIdx.y];
  const int k = f.k, nF = f.nF, p = nF - k;
  const int64_t tot = (int64_t)k * k;
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= tot) return;
  const int r = (int)(e % k), c = (int)(e / k);
  if (r < c) return;
  const T v = Zar[f.Z + (p + r) + (int64_t)(p + c) * nF];
  const int32_t* pm = perm + f.perm;
  const int32_t* rp = rowPos + f.rows;
  const int gr = pm[r], gc = pm[c];
  for (int i = 0; i < ncp; ++i) {
    const CellDesc cd = cells[f.cell[i]];
    const int x = rp[(int64_t)gr * ncp + i], y = rp[(int64_t)gc * ncp + i];
    if (x < 0 || y < 0) continue;
    const int hi_ = max(x, y), lo_ = min(x, y);
    Kar[cd.K + (cd.p + hi_) + (int64_t)(cd.p + lo_) * cd.n] = i == 0 ? v : T(0);
  }
}


// ---- row lists of faces and edges ------------------------------------------------
// Listing the rows on the host and uploading them was the longest wait of the
// level-0 plan (128^3: 15 million rows of 95232 faces, 38 ms); here a front is a
// block of 32 to 256 threads that walks its cells' lists, bound by the loads of
// the lists and of posb from L2.
struct DofGeom {
  int lc[3], sep;   // lowest cell holding the DOF, separator mask
};
__device__ __forceinline__ DofGeom dof_geom(const LevelGeom& geo, int g) {
  DofGeom d;
  const int z = g / (geo.n * geo.n), r = g - z * geo.n * geo.n;
  const int x[3] = {r % geo.n, r / geo.n, z};
  d.sep = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int q = x[i] / geo.s;
    const bool sd = x[i] == q * geo.s && (geo.wrap || x[i] != 0);
    d.lc[i] = sd ? (q == 0 ? geo.C - 1 : q - 1) : q;
    d.sep |= sd ? 1 << i : 0;
  }
  return d;
}
// corner of cell c (its three indices) relative to the DOF, -1 if its closure
// does not hold the DOF
__device__ __forceinline__ int corner_of(const LevelGeom& geo, const DofGeom& d, int c) {
  const int cc[3] = {c % geo.C, c / geo.C % geo.C, c / (geo.C * geo.C)};
  int q = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (cc[i] == d.lc[i]) continue;
    if (!((d.sep >> i) & 1) || cc[i] != (d.lc[i] + 1 == geo.C ? 0 : d.lc[i] + 1)) return -1;
    q |= 1 << i;
  }
  return q;
}

__global__ void k_cell_positions(LevelGeom geo, const CellDesc* __restrict__ cells,
                                 const int32_t* __restrict__ lists, int32_t* posb) {
  const CellDesc c = cells[blockIdx.x];
  const int32_t* b = lists + c.list + c.p;
  for (int t = threadIdx.x; t < c.n - c.p; t += blockDim.x) {
    const int g = b[t];
    const int q = corner_of(geo, dof_geom(geo, g), blockIdx.x);
    if (q >= 0) posb[(int64_t)g * 8 + q] = t;
  }
}

template <int NCP, bool FILL>
__global__ void k_skel_rows(LevelGeom geo, const RowFront* __restrict__ fronts,
                            const CellDesc* __restrict__ cells, const int32_t* __restrict__ lists,
                            const int32_t* __restrict__ posb, const uint8_t* __restrict__ alive,
                            int* nR, const int64_t* __restrict__ rowOff, int32_t* rowPos) {
  const RowFront f = fronts[blockIdx.x];
  const int nw = blockDim.x / 32, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  __shared__ int s_cnt[32];
  int32_t* out = FILL ? rowPos + rowOff[blockIdx.x] * NCP : nullptr;
  int64_t base = 0;   // rows so far (the same in every thread)
  const int low[3] = {f.cell[0] % geo.C, f.cell[0] / geo.C % geo.C, f.cell[0] / (geo.C * geo.C)};
  // pass -1: the front's own DOFs, from its first cell; pass i: the rows its
  // cell i adds
  for (int i = FILL ? -1 : 0; i < NCP; ++i) {
    const CellDesc c = cells[f.cell[max(i, 0)]];
    const int32_t* b = lists + c.list + c.p;
    const int nb = c.n - c.p;
    for (int t0 = 0; t0 < nb; t0 += blockDim.x) {
      const int t = t0 + threadIdx.x;
      bool take = false;
      int g = 0;
      DofGeom d{};
      if (t < nb) {
        g = b[t];
        d = dof_geom(geo, g);
        const bool own = d.sep == f.sep && d.lc[0] == low[0] && d.lc[1] == low[1] && d.lc[2] == low[2];
        if (i < 0) {
          take = own;
        } else if (!own && (!alive || alive[g])) {
          take = true;
          for (int j = 0; j < i; ++j) take = take && corner_of(geo, d, f.cell[j]) < 0;
        }
      }
      // the taken entries keep their order: place within the block
      const unsigned m = __ballot_sync(0xffffffffu, take);
      int before = __popc(m & ((1u << lane) - 1u)), all = __popc(m);
      if (nw > 1) {
        __syncthreads();
        if (lane == 0) s_cnt[warp] = all;
        __syncthreads();
        all = 0;
        for (int w = 0; w < nw; ++w) {
          before += w < warp ? s_cnt[w] : 0;
          all += s_cnt[w];
        }
      }
      if (FILL && take) {
        int32_t* o = out + (base + before) * NCP;
#pragma unroll
        for (int j = 0; j < NCP; ++j) {
          int pos = -1;
          if (j == max(i, 0)) {
            pos = t;
          } else if (j > i) {
            const int q = corner_of(geo, d, f.cell[j]);
            if (q >= 0) pos = posb[(int64_t)g * 8 + q];
          }
          o[j] = pos;
        }
      }
      base += all;
    }
  }
  if (!FILL && threadIdx.x == 0) nR[blockIdx.x] = (int)base;
}

}  // namespace

void cell_positions(const LevelGeom& geo, const CellDesc* d_cells, int ncell, const int32_t* lists,
                    int32_t* posb, cudaStream_t st) {
  if (ncell == 0) return;
  ProfScope ps("row_lists", st);
  k_cell_positions<<<ncell, 128, 0, st>>>(geo, d_cells, lists, posb);
  HIF_CHECK_LAUNCH();
}

void skel_rows(const LevelGeom& geo, const RowFront* d_fronts, int nf, int ncp,
               const CellDesc* d_cells, const int32_t* lists, const int32_t* posb,
               const uint8_t* alive, int mean_list, int* nR, const int64_t* rowOff, int32_t* rowPos,
               cudaStream_t st) {
  if (nf == 0) return;
  ProfScope ps("row_lists", st);
  // threads per front: one walk of the list in a few rounds
  const int th = mean_list <= 256 ? 32 : mean_list <= 1024 ? 128 : 256;
  auto go = [&](auto kern) {
    kern<<<nf, th, 0, st>>>(geo, d_fronts, d_cells, lists, posb, alive, nR, rowOff, rowPos);
    HIF_CHECK_LAUNCH();
  };
  if (ncp == 2) {
    if (rowPos) go(k_skel_rows<2, true>);
    else go(k_skel_rows<2, false>);
  } else {
    if (rowPos) go(k_skel_rows<4, true>);
    else go(k_skel_rows<4, false>);
  }
}

void stencil_coefficients(const double* a, const double* b, double b_const, int n, int periodic,
                          double* cpl, double* diag, int* d_bad, cudaStream_t st) {
  const int64_t N = (int64_t)n * n * n;
  ProfScope ps("stencil_coefficients", st, 0.0, 8.0 * N * (b ? 6.0 : 5.0));
  k_stencil<<<ceil_div(N, 256), 256, 0, st>>>(a, b, b_const, n, periodic, cpl, diag, d_bad);
  HIF_CHECK_LAUNCH();
}

void value_range(const double* a, int64_t cnt, unsigned long long* range, cudaStream_t st) {
  ProfScope ps("stencil_coefficients", st, 0.0, 8.0 * cnt);
  k_value_range<<<(int)std::min<int64_t>(304, (cnt + 255) / 256), 256, 0, st>>>(a, cnt, range);
  HIF_CHECK_LAUNCH();
}

template <typename T>
void assemble_level0(const CellDesc* d_cells, int ncell, const int32_t* lists, int n, int s,
                     int periodic, const double* cpl, const double* diag, T* Karena, int maxbox,
                     cudaStream_t st) {
  const size_t smem = (size_t)maxbox * sizeof(int);
  if (smem > 48 * 1024)
    HIF_CUDA_TRY(cudaFuncSetAttribute(k_assemble0<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
  ProfScope ps("assemble_level0", st);
  k_assemble0<T><<<ncell, 128, smem, st>>>(d_cells, lists, n, s, periodic, cpl, diag, Karena);
  HIF_CHECK_LAUNCH();
}

template <typename T>
void merge_children(const MergeDesc* d_par, const MergeDesc* h_par, int npar,
                    const CellDesc* d_child, const int32_t* maps, const T* Kchild, T* Kpar,
                    cudaStream_t st) {
  int nmax = 1;
  for (int i = 0; i < npar; ++i) nmax = std::max(nmax, h_par[i].n);
  const int nt = ceil_div(nmax, 64);
  for (int f0 = 0; f0 < npar; f0 += MAX_GRID_Y) {
    const int nb = std::min(MAX_GRID_Y, npar - f0);
    double by = 0;
    if (prof_enabled())
      for (int i = f0; i < f0 + nb; ++i) by += sizeof(T) * 0.5 * (double)h_par[i].n * (h_par[i].n + 1);
    ProfScope ps("merge_children", st, 0.0, by);
    k_merge<T><<<dim3(nt * (nt + 1) / 2, nb), 256, 0, st>>>(d_par + f0, d_child, maps, Kchild,
                                                            Kpar);
    HIF_CHECK_LAUNCH();
  }
}

template <typename T>
void skel_gather(const SkelDesc* d_f, const SkelDesc* h_f, int nf, int ncp,
                 const int32_t* rowPos, const CellDesc* d_cells, const T* Karena, T* Garena,
                 cudaStream_t st) {
  int64_t mx = 1;
  for (int i = 0; i < nf; ++i)
    mx = std::max<int64_t>(mx, (int64_t)ceil_div(h_f[i].nF + h_f[i].nR, GT) * ceil_div(h_f[i].nF, GT));
  for (int f0 = 0; f0 < nf; f0 += MAX_GRID_Y) {
    const int nb = std::min(MAX_GRID_Y, nf - f0);
    double by = 0;
    if (prof_enabled())
      for (int i = f0; i < f0 + nb; ++i) by += sizeof(T) * (double)(h_f[i].nF + h_f[i].nR) * h_f[i].nF;
    ProfScope ps("skel_gather", st, 0.0, by);
    k_skel_gather<T><<<dim3((unsigned)mx, nb), 256, 0, st>>>(d_f + f0, ncp, rowPos, d_cells,
                                                             Karena, Garena);
    HIF_CHECK_LAUNCH();
  }
}

template <typename T>
void skel_permute(const SkelDesc* d_f, const SkelDesc* h_f, int nf, const int32_t* perm,
                  const T* Garena, T* Zarena, cudaStream_t st) {
  int64_t mx = 1;
  for (int i = 0; i < nf; ++i) mx = std::max<int64_t>(mx, (int64_t)h_f[i].nF * h_f[i].nF);
  for (int f0 = 0; f0 < nf; f0 += MAX_GRID_Y) {
    const int nb = std::min(MAX_GRID_Y, nf - f0);
    ProfScope ps("skel_permute", st);
    k_skel_permute<T><<<dim3(ceil_div(mx, 256), nb), 256, 0, st>>>(d_f + f0, perm, Garena, Zarena);
    HIF_CHECK_LAUNCH();
  }
}

template <typename T>
void skel_writeback(const SkelDesc* d_f, const SkelDesc* h_f, int nf, int ncp,
                    const int32_t* rowPos, const int32_t* perm, const CellDesc* d_cells,
                    const T* Zarena, T* Karena, cudaStream_t st) {
  int64_t mx = 1;
  for (int i = 0; i < nf; ++i) mx = std::max<int64_t>(mx, (int64_t)h_f[i].k * h_f[i].k);
  for (int f0 = 0; f0 < nf; f0 += MAX_GRID_Y) {
    const int nb = std::min(MAX_GRID_Y, nf - f0);
    ProfScope ps("skel_writeback", st);
    k_skel_writeback<T><<<dim3(ceil_div(mx, 256), nb), 256, 0, st>>>(d_f + f0, ncp, rowPos, perm,
                                                                     d_cells, Zarena, Karena);
    HIF_CHECK_LAUNCH();
  }
}

#define HIF_INST(T)                                                                          \
  template void assemble_level0<T>(const CellDesc*, int, const int32_t*, int, int, int,     \
                                   const double*, const double*, T*, int, cudaStream_t);    \
  template void merge_children<T>(const MergeDesc*, const MergeDesc*, int, const CellDesc*, \
                                  const int32_t*, const T*, T*, cudaStream_t);              \
  template void skel_gather<T>(const SkelDesc*, const SkelDesc*, int, int, const int32_t*,  \
                               const CellDesc*, const T*, T*, cudaStream_t);                \
  template void skel_permute<T>(const SkelDesc*, const SkelDesc*, int, const int32_t*,      \
                                const T*, T*, cudaStream_t);                                \
  template void skel_writeback<T>(const SkelDesc*, const SkelDesc*, int, int,               \
                                  const int32_t*, const int32_t*, const CellDesc*,          \
                                  const T*, T*, cudaStream_t);
HIF_INST(float)
HIF_INST(double)
#undef HIF_INST

}  // namespace hif
