// Kernels that build the base-case structures once per grid: branch
// admittances, the bus admittance diagonal, the B'/B'' values (Sec. III.B:
// the diagonal .BIJ on the vertex, the off-diagonal .BIJ on the edge) and the
// level-scheduled numeric factorisation of the base-case matrix that
// preconditions every scenario (Sec. IV.B, eq. (6)).
#include "common.cuh"

namespace gpcg {

// y = 1/(r + jx) = g + j b_y; weights of B' (1/x) and B'' (x/(r^2+x^2)).
__global__ void branch_params_kernel(int m, const double* __restrict__ r,
                                     const double* __restrict__ x, double* g, double* by,
                                     double* wP, double* wQ) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m) return;
  double rr = r[e], xx = x[e];
  double d = rr * rr + xx * xx;
  g[e] = rr / d;
  by[e] = -xx / d;
  wP[e] = 1.0 / xx;
  wQ[e] = xx / d;
}

// Y_ii = sum over incident branches of (y + j b_sh/2), times c^2 at the
// from end of a transformer (c = 1 / turns ratio: the pi-model sees V_i c),
// summed in the fixed order of the bus adjacency lists.
__global__ void ybus_diag_kernel(int n, const int32_t* __restrict__ adj_ptr,
                                 const int32_t* __restrict__ adj_br,
                                 const int32_t* __restrict__ from, const double* __restrict__ cf,
                                 const double* __restrict__ g, const double* __restrict__ by,
                                 const double* __restrict__ b_sh, double2* ydiag) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double G = 0.0, B = 0.0;
  for (int k = adj_ptr[i]; k < adj_ptr[i + 1]; ++k) {
    int e = adj_br[k];
    const double c2 = from[e] == i ? cf[e] * cf[e] : 1.0;
    G += c2 * g[e];
    B += c2 * (by[e] + 0.5 * b_sh[e]);
  }
  ydiag[i] = make_double2(G, B);
}

// Values of a grounded sum of branch terms w v v^T, v = c e_from - e_to
// (c = 1 for every branch when cf is null: a weighted Laplacian), on its CSR
// pattern: one thread per matrix row walks the bus's incident branches in a
// fixed order.  The diagonal collects every incident branch (also those to
// buses without a row), w c^2 at a from end and w at a to end; each
// neighbour with a row receives -w c in its slot.
__global__ void laplacian_values_kernel(int nrows, const int32_t* __restrict__ bus_of_row,
                                        const int32_t* __restrict__ row_of_bus,
                                        const int32_t* __restrict__ adj_ptr,
                                        const int32_t* __restrict__ adj_idx,
                                        const int32_t* __restrict__ adj_br,
                                        const double* __restrict__ w,
                                        const int32_t* __restrict__ from,
                                        const double* __restrict__ cf,
                                        const int32_t* __restrict__ a_ptr,
                                        const int32_t* __restrict__ a_idx, double* a_val,
                                        int32_t* err) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nrows) return;
  int b = bus_of_row[i];
  int s = a_ptr[i], e_ = a_ptr[i + 1];
  for (int k = s; k < e_; ++k) a_val[k] = 0.0;
  double diag = 0.0;
  for (int k = adj_ptr[b]; k < adj_ptr[b + 1]; ++k) {
    const int e = adj_br[k];
    double we = w[e];
    if (cf) {
      diag += from[e] == b ? we * cf[e] * cf[e] : we;
      we *= cf[e];
    } else {
      diag += we;
    }
    int c = row_of_bus[adj_idx[k]];
    if (c < 0) continue;
    int lo = s, hi = e_ - 1, pos = -1;
    while (lo <= hi) {
      int mid = (lo + hi) >> 1;
      int v = a_idx[mid];
      if (v == c) { pos = mid; break; }
      if (v < c) lo = mid + 1; else hi = mid - 1;
    }
    if (pos < 0) { atomicExch(err, 1); continue; }
    a_val[pos] -= we;
  }
  int lo = s, hi = e_ - 1, pos = -1;
  while (lo <= hi) {
    int mid = (lo + hi) >> 1;
    int v = a_idx[mid];
    if (v == i) { pos = mid; break; }
    if (v < i) lo = mid + 1; else hi = mid - 1;
  }
  if (pos < 0) { atomicExch(err, 1); return; }
  a_val[pos] += diag;
}

// The row a bus without one would have in a matrix of branch terms w v v^T
// (v = c e_from - e_to; cf null: c = 1), for every bus: per adjacency entry
// the neighbour's row (-1: none) and -w c, and per bus the diagonal, summed
// in the same order and form as laplacian_values_kernel.
__global__ void ext_rows_kernel(int n, const int32_t* __restrict__ adj_ptr,
                                const int32_t* __restrict__ adj_idx,
                                const int32_t* __restrict__ adj_br,
                                const int32_t* __restrict__ from, const double* __restrict__ cf,
                                const double* __restrict__ w,
                                const int32_t* __restrict__ row_of_bus, int32_t* xrow,
                                double* xval, float* xval32, double* xdiag, float* xdiag32) {
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  double diag = 0.0;
  for (int k = adj_ptr[b]; k < adj_ptr[b + 1]; ++k) {
    const int e = adj_br[k];
    double we = w[e];
    if (cf) {
      diag += from[e] == b ? we * cf[e] * cf[e] : we;
      we *= cf[e];
    } else {
      diag += we;
    }
    xrow[k] = row_of_bus[adj_idx[k]];
    xval[k] = -we;
    xval32[k] = (float)-we;
  }
  xdiag[b] = diag;
  xdiag32[b] = (float)diag;
}

void launch_ext_rows(cudaStream_t st, int n, const int32_t* adj_ptr, const int32_t* adj_idx,
                     const int32_t* adj_br, const int32_t* from, const double* cf,
                     const double* w, const int32_t* row_of_bus, int32_t* xrow, double* xval,
                     float* xval32, double* xdiag, float* xdiag32) {
  if (n > 0)
    ext_rows_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, adj_ptr, adj_idx, adj_br, from, cf, w,
                                                     row_of_bus, xrow, xval, xval32, xdiag,
                                                     xdiag32);
}

__device__ __forceinline__ double csr_lookup(const int32_t* idx, const double* val, int s,
                                             int e, int col) {
  int lo = s, hi = e - 1;
  while (lo <= hi) {
    int mid = (lo + hi) >> 1;
    int v = idx[mid];
    if (v == col) return val[mid];
    if (v < col) lo = mid + 1; else hi = mid - 1;
  }
  return 0.0;
}

// Incomplete Cholesky on the pattern of L, rows of one level at a time (all
// rows a row depends on sit in lower levels):
//   L_ij = (A_ij - sum_{k<j} L_ik L_jk) / L_jj,   L_ii = sqrt(A_ii - sum L_ik^2),
// the sums running over the columns both rows hold.  With the complete
// symbolic pattern this is the exact Cholesky factor.
__global__ void ic_level_kernel(int row0, int row1, const int32_t* __restrict__ a_ptr,
                                const int32_t* __restrict__ a_idx,
                                const double* __restrict__ a_val,
                                const int32_t* __restrict__ l_ptr,
                                const int32_t* __restrict__ l_idx, double* l_val,
                                int32_t* err) {
  int i = row0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= row1) return;
  int ls = l_ptr[i], le = l_ptr[i + 1];
  for (int k = ls; k < le; ++k) {
    int j = l_idx[k];
    double s = csr_lookup(a_idx, a_val, a_ptr[i], a_ptr[i + 1], j);
    // merge row i (entries before k) with row j (off-diagonal entries)
    int p = ls, q = l_ptr[j], qe = l_ptr[j + 1] - 1;
    while (p < k && q < qe) {
      int ci = l_idx[p], cj = l_idx[q];
      if (ci == cj) { s -= l_val[p] * l_val[q]; ++p; ++q; }
      else if (ci < cj) ++p;
      else ++q;
    }
    if (j < i) {
      l_val[k] = s / l_val[l_ptr[j + 1] - 1];
    } else {
      if (!(s > 0.0)) { atomicExch(err, 2); s = 1.0; }
      l_val[k] = sqrt(s);
    }
  }
}

// The narrow levels [lev0, lev1) in one launch of one CTA, a warp per row, for
// the adjoint, which factorises on every call: a launch per level (67 on a
// 2,000-bus grid) and a thread walking both rows of every product one entry at a
// time took most of a re-factorisation.  A context's own factor keeps the sums
// in row order (ic_level_kernel): the last bits of the base case and of the
// FP32 factor decide the verdicts of scenarios that have no solution.  The row's
// entries are computed in order; the sum over the columns rows i and j share has
// its terms spread over the warp (each looks the column of row j up in row i).
constexpr int IC_NARROW = 512;  // rows of a level, at most
__global__ void __launch_bounds__(1024)
    ic_narrow_kernel(const int32_t* __restrict__ lev_ptr, int lev0, int lev1,
                     const int32_t* __restrict__ a_ptr, const int32_t* __restrict__ a_idx,
                     const double* __restrict__ a_val, const int32_t* __restrict__ l_ptr,
                     const int32_t* __restrict__ l_idx, double* l_val, int32_t* err) {
  const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
  for (int lev = lev0; lev < lev1; ++lev) {
    const int r1 = lev_ptr[lev + 1];
    for (int i = lev_ptr[lev] + warp; i < r1; i += 32) {
      const int ls = l_ptr[i], le = l_ptr[i + 1];
      for (int k = ls; k < le; ++k) {
        const int j = l_idx[k], q0 = l_ptr[j], q1 = l_ptr[j + 1] - 1;
        double s = 0.0;
        for (int q = q0 + wl; q < q1; q += 32) {
          const int c = l_idx[q];
          int lo = ls, hi = k;  // row i's entries before k
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (l_idx[mid] < c) lo = mid + 1; else hi = mid;
          }
          if (lo < k && l_idx[lo] == c) s = fma(l_val[lo], l_val[q], s);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (wl == 0) {
          s = csr_lookup(a_idx, a_val, a_ptr[i], a_ptr[i + 1], j) - s;
          if (j < i) {
            l_val[k] = s / l_val[q1];
          } else {
            if (!(s > 0.0)) { atomicExch(err, 2); s = 1.0; }
            l_val[k] = sqrt(s);
          }
        }
        __syncwarp();
      }
    }
    __syncthreads();
  }
}

__global__ void scatter_kernel(int nnz, const int32_t* __restrict__ map,
                               const double* __restrict__ src, double* dst) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nnz) dst[map[k]] = src[k];
}

__global__ void to_float_kernel(int n, const double* __restrict__ src, float* dst) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) dst[k] = (float)src[k];
}

__global__ void gather_diag_kernel(int n, const int32_t* __restrict__ pos,
                                   const double* __restrict__ a_val, double* d) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) d[k] = a_val[pos[k]];
}

__global__ void gather_int_kernel(int n, const int32_t* __restrict__ idx,
                                  const int32_t* __restrict__ src, int32_t* dst) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) dst[k] = src[idx[k]];
}

// ---------------------------------------------------------------- launchers
static inline int nblk(int n, int b) { return (n + b - 1) / b; }

void launch_branch_params(cudaStream_t st, int m, const double* r, const double* x, double* g,
                          double* by, double* wP, double* wQ) {
  if (m) branch_params_kernel<<<nblk(m, 256), 256, 0, st>>>(m, r, x, g, by, wP, wQ);
}
void launch_ybus_diag(cudaStream_t st, int n, const int32_t* adj_ptr, const int32_t* adj_br,
                      const int32_t* from, const double* cf, const double* g, const double* by,
                      const double* b_sh, double2* ydiag) {
  if (n)
    ybus_diag_kernel<<<nblk(n, 256), 256, 0, st>>>(n, adj_ptr, adj_br, from, cf, g, by, b_sh,
                                                   ydiag);
}
void launch_laplacian_values(cudaStream_t st, int nrows, const int32_t* bus_of_row,
                             const int32_t* row_of_bus, const int32_t* adj_ptr,
                             const int32_t* adj_idx, const int32_t* adj_br, const double* w,
                             const int32_t* from, const double* cf, const int32_t* a_ptr,
                             const int32_t* a_idx, double* a_val, int32_t* err) {
  if (nrows)
    laplacian_values_kernel<<<nblk(nrows, 128), 128, 0, st>>>(
        nrows, bus_of_row, row_of_bus, adj_ptr, adj_idx, adj_br, w, from, cf, a_ptr, a_idx,
        a_val, err);
}
void launch_ic_level(cudaStream_t st, int row0, int row1, const int32_t* a_ptr,
                     const int32_t* a_idx, const double* a_val, const int32_t* l_ptr,
                     const int32_t* l_idx, double* l_val, int32_t* err) {
  int n = row1 - row0;
  if (n > 0)
    ic_level_kernel<<<nblk(n, 128), 128, 0, st>>>(row0, row1, a_ptr, a_idx, a_val, l_ptr,
                                                  l_idx, l_val, err);
}
void launch_ic_narrow(cudaStream_t st, const int32_t* lev_ptr, int lev0, int lev1,
                      const int32_t* a_ptr, const int32_t* a_idx, const double* a_val,
                      const int32_t* l_ptr, const int32_t* l_idx, double* l_val, int32_t* err) {
  if (lev1 > lev0)
    ic_narrow_kernel<<<1, 1024, 0, st>>>(lev_ptr, lev0, lev1, a_ptr, a_idx, a_val, l_ptr, l_idx,
                                         l_val, err);
}
int ic_narrow_rows() { return IC_NARROW; }
void launch_scatter(cudaStream_t st, int nnz, const int32_t* map, const double* src,
                    double* dst) {
  if (nnz) scatter_kernel<<<nblk(nnz, 256), 256, 0, st>>>(nnz, map, src, dst);
}
void launch_to_float(cudaStream_t st, int n, const double* src, float* dst) {
  if (n) to_float_kernel<<<nblk(n, 256), 256, 0, st>>>(n, src, dst);
}
void launch_gather_diag(cudaStream_t st, int n, const int32_t* pos, const double* a_val,
                        double* d) {
  if (n) gather_diag_kernel<<<nblk(n, 256), 256, 0, st>>>(n, pos, a_val, d);
}
void launch_gather_int(cudaStream_t st, int n, const int32_t* idx, const int32_t* src,
                       int32_t* dst) {
  if (n) gather_int_kernel<<<nblk(n, 256), 256, 0, st>>>(n, idx, src, dst);
}

}  // namespace gpcg

namespace gpcg {

// dst[k] = csr[src[k]] (0 where src[k] < 0), in FP64 and FP32.
__global__ void gather_val_kernel(int n, const int32_t* __restrict__ src,
                                  const double* __restrict__ csr, double* dst, float* dst32) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int s = src[k];
  const double v = s >= 0 ? csr[s] : 0.0;
  dst[k] = v;
  dst32[k] = (float)v;
}

__global__ void inv_diag_kernel(int n, const int32_t* __restrict__ pos,
                                const double* __restrict__ l_val, double* inv, float* inv32) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double d = 1.0 / l_val[pos[i]];
  inv[i] = d;
  inv32[i] = (float)d;
}

// Per-slot branch admittance of the mismatch adjacency (0 on padding), as
// pairs (gb) or in two arrays.
__global__ void adj_values_kernel(int n, const int32_t* __restrict__ br,
                                  const double* __restrict__ cf,
                                  const double* __restrict__ g, const double* __restrict__ by,
                                  double2* gb, double* ag, double* ab) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int e = br[k];
  // Y_ij = -c y for either end (c = 1 / turns ratio)
  const double yg = e >= 0 ? cf[e] * g[e] : 0.0, yb = e >= 0 ? cf[e] * by[e] : 0.0;
  if (gb) {
    gb[k] = make_double2(yg, yb);
  } else {
    ag[k] = yg;
    ab[k] = yb;
  }
}

// The admittances the branch flows take (DevGrid::ybr).
__global__ void flow_values_kernel(int m, const double* __restrict__ cf,
                                   const double* __restrict__ g, const double* __restrict__ by,
                                   double2* ybr) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const double c = cf[k];
  ybr[2 * (size_t)k] = make_double2(g[k] * c * c, g[k] * c);
  ybr[2 * (size_t)k + 1] = make_double2(by[k] * c, g[k]);
}
void launch_flow_values(cudaStream_t st, int m, const double* cf, const double* g,
                        const double* by, double2* ybr) {
  if (m > 0) flow_values_kernel<<<(m + 255) / 256, 256, 0, st>>>(m, cf, g, by, ybr);
}

__global__ void gather_pair_kernel(int n, const int4* __restrict__ md,
                                   const double2* __restrict__ src, double2* dst) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) dst[k] = src[md[k].x];
}
void launch_gather_pair(cudaStream_t st, int n, const int4* md, const double2* src,
                        double2* dst) {
  if (n > 0) gather_pair_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, md, src, dst);
}

void launch_gather_val(cudaStream_t st, int n, const int32_t* src, const double* csr, double* dst,
                       float* dst32) {
  if (n > 0) gather_val_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, src, csr, dst, dst32);
}
void launch_inv_diag(cudaStream_t st, int n, const int32_t* pos, const double* l_val, double* inv,
                     float* inv32) {
  if (n > 0) inv_diag_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, pos, l_val, inv, inv32);
}
// X = inverse of the factor's tail block L_tt (rows and columns
// [t0, t0 + nt) of L, lower triangular): column c of X by forward
// substitution of L_tt x = e_c, one thread per column (as many CTAs as leave no
// thread two of the serial chains), in FP64.  Written
// column-major (xc[c nt + i] = X_ic) and row-major (xr[i nt + c] = X_ic),
// zeros above the diagonal, in FP64 (xr optional) and FP32.
// With lsc (the scaled factor Ls = L D^-1) the block inverted is the one
// the FP16 storage represents: L_ij = fp16(Ls_ij) L_jj.
__global__ void tail_inverse_kernel(int t0, int nt, const int32_t* __restrict__ l_ptr,
                                    const int32_t* __restrict__ l_idx,
                                    const double* __restrict__ l_val,
                                    const double* __restrict__ lsc, double* xc, double* xr,
                                    float* xc32, float* xr32) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < nt) {
    // xc holds the column in FP64 while it is built (its earlier entries
    // are the unknowns solved before)
    for (int i = 0; i < nt; ++i) {
      double v = 0.0;
      if (i >= c) {
        const int R = t0 + i, e0 = l_ptr[R], e1 = l_ptr[R + 1] - 1;  // diagonal last
        double sum = (i == c) ? 1.0 : 0.0;
        for (int e = e0; e < e1; ++e) {
          const int jg = l_idx[e], j = jg - t0;
          if (j < c) continue;
          const double lij =
              lsc ? (double)__half2float(__double2half(lsc[e])) * l_val[l_ptr[jg + 1] - 1]
                  : l_val[e];
          sum -= lij * xc[(size_t)c * nt + j];
        }
        v = sum / l_val[e1];
      }
      xc[(size_t)c * nt + i] = v;
      if (xr) xr[(size_t)i * nt + c] = v;
      xc32[(size_t)c * nt + i] = (float)v;
      xr32[(size_t)i * nt + c] = (float)v;
    }
  }
}

// The same for the adjoint (see ic_narrow_kernel): a warp per column, the row's
// terms spread over its threads (a thread per column waits for the loads of each
// term: about 1 ms for 232 rows).
constexpr int TI_WARPS = 4;
__global__ void __launch_bounds__(32 * TI_WARPS)
    tail_inverse_warp_kernel(int t0, int nt, const int32_t* __restrict__ l_ptr,
                             const int32_t* __restrict__ l_idx,
                             const double* __restrict__ l_val, double* xc, double* xr,
                             float* xc32, float* xr32) {
  __shared__ double col[TI_WARPS][TAIL_ROWS];
  const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
  const int c = blockIdx.x * TI_WARPS + warp;
  if (c >= nt) return;
  double* x = col[warp];
  for (int i = wl; i < c; i += 32) x[i] = 0.0;
  for (int i = c; i < nt; ++i) {
    const int R = t0 + i, e0 = l_ptr[R], e1 = l_ptr[R + 1] - 1;  // diagonal last
    double s = 0.0;
    for (int e = e0 + wl; e < e1; e += 32) {
      const int j = l_idx[e] - t0;
      if (j < c) continue;
      s = fma(l_val[e], x[j], s);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (wl == 0) x[i] = ((i == c ? 1.0 : 0.0) - s) / l_val[e1];
    __syncwarp();
  }
  for (int i = wl; i < nt; i += 32) {
    const double v = x[i];
    xc[(size_t)c * nt + i] = v;
    xr[(size_t)i * nt + c] = v;
    xc32[(size_t)c * nt + i] = (float)v;
    xr32[(size_t)i * nt + c] = (float)v;
  }
}

void launch_tail_inverse(cudaStream_t st, int t0, int nt, const int32_t* l_ptr,
                         const int32_t* l_idx, const double* l_val, const double* lsc, double* xc,
                         double* xr, float* xc32, float* xr32) {
  if (nt > 0)
    tail_inverse_kernel<<<(nt + 127) / 128, 128, 0, st>>>(t0, nt, l_ptr, l_idx, l_val, lsc, xc, xr,
                                                       xc32, xr32);
}
void launch_tail_inverse_warp(cudaStream_t st, int t0, int nt, const int32_t* l_ptr,
                              const int32_t* l_idx, const double* l_val, double* xc, double* xr,
                              float* xc32, float* xr32) {
  if (nt > 0)
    tail_inverse_warp_kernel<<<(nt + TI_WARPS - 1) / TI_WARPS, 32 * TI_WARPS, 0, st>>>(
        t0, nt, l_ptr, l_idx, l_val, xc, xr, xc32, xr32);
}

void launch_adj_values(cudaStream_t st, int n, const int32_t* br, const double* cf,
                       const double* g, const double* by, double2* gb, double* ag, double* ab) {
  if (n > 0) adj_values_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, br, cf, g, by, gb, ag, ab);
}

}  // namespace gpcg

namespace gpcg {

// Scaled factor for FP16 storage: L = Ls D, D = diag(L); Ls_ij = L_ij / L_jj
// (unit diagonal), and 1 / L_ii^2 for the back substitution.
__global__ void scale_factor_kernel(int n, const int32_t* __restrict__ l_ptr,
                                    const int32_t* __restrict__ l_idx,
                                    const double* __restrict__ l_val, double* lsc, double* inv_d2,
                                    float* inv_d2_32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int k = l_ptr[i]; k < l_ptr[i + 1]; ++k) {
    const int j = l_idx[k];
    lsc[k] = l_val[k] / l_val[l_ptr[j + 1] - 1];
  }
  const double d = l_val[l_ptr[i + 1] - 1];
  inv_d2[i] = 1.0 / (d * d);
  inv_d2_32[i] = (float)(1.0 / (d * d));
}

__global__ void gather_half_kernel(int n, const int32_t* __restrict__ src,
                                   const double* __restrict__ v, __half* dst) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int s = src[k];
  dst[k] = __double2half(s >= 0 ? v[s] : 0.0);
}

void launch_scale_factor(cudaStream_t st, int n, const int32_t* l_ptr, const int32_t* l_idx,
                         const double* l_val, double* lsc, double* inv_d2, float* inv_d2_32) {
  if (n > 0)
    scale_factor_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, l_ptr, l_idx, l_val, lsc, inv_d2,
                                                         inv_d2_32);
}
void launch_gather_half(cudaStream_t st, int n, const int32_t* src, const double* v, __half* dst) {
  if (n > 0) gather_half_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, src, v, dst);
}

}  // namespace gpcg

// ------------------------------------------------------- branch columns
namespace gpcg {

// The rows of L^-1 v for a vector v with entries at rows a and b (-1: none):
// both ends' chains of elimination-tree ancestors, merged in ascending order
// (parents have larger row numbers).  Calls visit(row) for each.
template <typename F>
__device__ __forceinline__ void walk_ancestors(const int32_t* __restrict__ parent, int a, int b,
                                               F visit) {
  while (a >= 0 || b >= 0) {
    int& next = b < 0 || (a >= 0 && a < b) ? a : b;
    visit(next);
    next = parent[next];
    if (a == b && a >= 0) {  // the chains have met: one from here on
      for (; a >= 0; a = parent[a]) visit(a);
      return;
    }
  }
}

__global__ void branch_count_kernel(int m, const int32_t* __restrict__ f,
                                    const int32_t* __restrict__ t,
                                    const int32_t* __restrict__ row_of_bus,
                                    const int32_t* __restrict__ parent, int32_t* cnt) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= m) return;
  int k = 0;
  walk_ancestors(parent, row_of_bus[f[l]], row_of_bus[t[l]], [&](int) { ++k; });
  cnt[l] = k;
}

// One thread per branch: the rows, L^-1 v and L^-1 v_m by forward
// substitution over them (column-oriented: every entry of a column of L on
// the path lies on the path), and the branch's scalars.  13,500 branches of a
// 10,000-bus grid have about 60 rows each.
__global__ void branch_cols_kernel(int m, const int32_t* __restrict__ f,
                                   const int32_t* __restrict__ t,
                                   const int32_t* __restrict__ row_of_bus,
                                   const int32_t* __restrict__ parent,
                                   const int32_t* __restrict__ ucol,
                                   const double* __restrict__ uval,
                                   const int32_t* __restrict__ uoptr,
                                   const int32_t* __restrict__ uocol,
                                   const double* __restrict__ uoval, int n,
                                   const double* __restrict__ inv_diag,
                                   const double* __restrict__ w, const double* __restrict__ cf,
                                   const int32_t* __restrict__ pre,
                                   const int32_t* __restrict__ br_lo,
                                   const int32_t* __restrict__ br_cnt,
                                   const int32_t* __restrict__ ptr, int32_t* row, double* fv,
                                   double* fm, double* sc) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= m) return;
  const int ra = row_of_bus[f[l]], rb = row_of_bus[t[l]];
  const int p0 = ptr[l], p1 = ptr[l + 1];
  {
    int k = p0;
    walk_ancestors(parent, ra, rb, [&](int i) { row[k++] = i; });
  }
  const double c = cf ? cf[l] : 1.0;
  // a bridge: the island's end is not part of the main island's system
  const int lo = br_lo[l], cn = br_cnt[l];
  const double ca = ra >= 0 && !in_island(pre[f[l]], lo, cn) ? c : 0.0;
  const double cb = rb >= 0 && !in_island(pre[t[l]], lo, cn) ? -1.0 : 0.0;
  for (int e = p0; e < p1; ++e) {
    const int i = row[e];
    fv[e] = i == ra ? c : i == rb ? -1.0 : 0.0;
    fm[e] = i == ra ? ca : i == rb ? cb : 0.0;
  }
  double vy = 0.0, my = 0.0, vv = 0.0;
  for (int e = p0; e < p1; ++e) {
    const int j = row[e];
    const double a = fv[e] * inv_diag[j], b = fm[e] * inv_diag[j];
    fv[e] = a;
    fm[e] = b;
    vy = fma(a, b, vy);
    my = fma(b, b, my);
    vv = fma(a, a, vv);
    auto spread = [&](int k, double v) {
      int x = e + 1, y = p1 - 1;  // row k's place: every k is an ancestor of j
      while (x < y) {
        const int mid = (x + y) >> 1;
        if (row[mid] < k) x = mid + 1; else y = mid;
      }
      fv[x] = fma(-v, a, fv[x]);
      fm[x] = fma(-v, b, fm[x]);
    };
    for (int s = 0; s < KU; ++s) {
      const int k = ucol[(size_t)j * KU + s];
      if (k < n) spread(k, uval[(size_t)j * KU + s]);
    }
    for (int s = uoptr[j]; s < uoptr[j + 1]; ++s) spread(uocol[s], uoval[s]);
  }
  double* o = sc + (size_t)l * SC_N;
  o[SC_VY] = vy;
  o[SC_MY] = my;
  o[SC_VM2] = ca * ca + cb * cb;
  o[SC_CA] = ca;
  o[SC_CB] = cb;
  o[SC_W] = w[l];
  o[SC_VV] = vv;
}

// L^-1 c_b of the buses with rows in bptr (BusCols), one thread per bus; the
// couplings from the bus's adjacency (xptr, xrow, xval).
__global__ void bus_cols_kernel(int nb, const int32_t* __restrict__ xptr,
                                const int32_t* __restrict__ xrow,
                                const double* __restrict__ xval, const int32_t* __restrict__ ucol,
                                const double* __restrict__ uval,
                                const int32_t* __restrict__ uoptr,
                                const int32_t* __restrict__ uocol,
                                const double* __restrict__ uoval, int n,
                                const double* __restrict__ inv_diag,
                                const int32_t* __restrict__ ptr, const int32_t* __restrict__ row,
                                double* f, double* ff) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  const int p0 = ptr[b], p1 = ptr[b + 1];
  double s2 = 0.0;
  if (p0 < p1) {
    auto place = [&](int from, int k) {
      int x = from, y = p1 - 1;
      while (x < y) {
        const int mid = (x + y) >> 1;
        if (row[mid] < k) x = mid + 1; else y = mid;
      }
      return x;
    };
    for (int e = p0; e < p1; ++e) f[e] = 0.0;
    for (int e = xptr[b]; e < xptr[b + 1]; ++e)
      if (xrow[e] >= 0) f[place(p0, xrow[e])] += xval[e];
    for (int e = p0; e < p1; ++e) {
      const int j = row[e];
      const double a = f[e] * inv_diag[j];
      f[e] = a;
      s2 = fma(a, a, s2);
      for (int s = 0; s < KU; ++s) {
        const int k = ucol[(size_t)j * KU + s];
        if (k < n) f[place(e + 1, k)] -= uval[(size_t)j * KU + s] * a;
      }
      for (int s = uoptr[j]; s < uoptr[j + 1]; ++s) f[place(e + 1, uocol[s])] -= uoval[s] * a;
    }
  }
  ff[b] = s2;
}
void launch_bus_cols(cudaStream_t st, int nb, const int32_t* xptr, const int32_t* xrow,
                     const double* xval, const Ell<double>& U, int n, const double* inv_diag,
                     const int32_t* ptr, const int32_t* row, double* f, double* ff) {
  if (nb > 0)
    bus_cols_kernel<<<nblk(nb, 128), 128, 0, st>>>(nb, xptr, xrow, xval, U.col, U.val, U.optr,
                                                   U.ocol, U.oval, n, inv_diag, ptr, row, f, ff);
}

void launch_branch_count(cudaStream_t st, int m, const int32_t* f, const int32_t* t,
                         const int32_t* row_of_bus, const int32_t* parent, int32_t* cnt) {
  if (m > 0) branch_count_kernel<<<nblk(m, 128), 128, 0, st>>>(m, f, t, row_of_bus, parent, cnt);
}
void launch_branch_cols(cudaStream_t st, int m, const int32_t* f, const int32_t* t,
                        const int32_t* row_of_bus, const int32_t* parent, const Ell<double>& U,
                        int n, const double* inv_diag, const double* w, const double* cf,
                        const int32_t* pre, const int32_t* br_lo, const int32_t* br_cnt,
                        const int32_t* ptr, int32_t* row, double* fv, double* fm, double* sc) {
  if (m > 0)
    branch_cols_kernel<<<nblk(m, 128), 128, 0, st>>>(m, f, t, row_of_bus, parent, U.col, U.val,
                                                     U.optr, U.ocol, U.oval, n, inv_diag, w, cf,
                                                     pre, br_lo, br_cnt, ptr, row, fv, fm, sc);
}

}  // namespace gpcg
