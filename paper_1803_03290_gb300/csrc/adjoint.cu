// The overload-penalty adjoint over N-1 scenarios (DC model of eq. (4)).
//
// For scenario s (outage l): theta_s = B'_s^{-1} R_s P with B'_s the base
// matrix (weights b) minus the outaged branch's four-element change
// (Sec. IV.B), islands removed and their injection re-dispatched
// (Sec. IV.C, weights frozen); flows f = b (theta_i - theta_j);
// L = sum softplus(|f|/rating - 1)^2.  With g = dL/df the adjoint is one more
// solve with the symmetric B'_s, lambda_s = B'_s^{-1} A^T diag(b_s) g_s, and
//   dL/dP   = sum_s R_s^T lambda_s,
//   dL/db_k = sum_s [ g_ks (A theta_s)_k - (A lambda_s)_k (A theta_s)_k ].
// Both solves are the batched base-preconditioned PCG of the N-1 screen, in its
// reduced form (reduced.cuh) with the complete factor.
// Tiles are dealt to CTAs statically; each CTA accumulates its scenarios'
// terms in its own slot and a second kernel sums the slots in a fixed order,
// so the gradients are bitwise reproducible.
#include "reduced.cuh"

namespace gpcg {

struct AdjParams {
  const double* P = nullptr;   // [n] injections, internal bus order
  const double* b = nullptr;   // [m] branch susceptances
  double* gP = nullptr;        // [slots][n] per-slot sums (internal order)
  double* gb = nullptr;        // [slots][m]
  double* loss = nullptr;      // [slots]
  double* g = nullptr;         // [slots][m][2] dL/df of the slot's scenarios
};

// Penalty phi(F) = softplus(u)^2, u = |F| / rating - 1, and its derivative
// 2 softplus(u) sigmoid(u) sign(F) / rating (odd in F).  Both follow from
// e = exp(-|u|): softplus = max(u, 0) + log1p(e), sigmoid = 1 / (1 + e) or
// e / (1 + e).  An exponential, a logarithm and a division are about 75 FP64
// instructions, more than the rest of a branch's work together, so they are
// evaluated once per branch and scenario and the derivative is kept (four
// evaluations, with the reduced solves and the slot sums below: a call for all
// 2,700 outages of 2,000 buses 16.6 -> 5.6 ms).
__device__ __forceinline__ double penalty(double F, double inv_rating, double& grad) {
  const double u = fma(fabs(F), inv_rating, -1.0);
  const double e = exp(-fabs(u)), d = 1.0 / (1.0 + e);
  const double s = fmax(u, 0.0) + log1p(e);
  grad = copysign(2.0 * s * (u > 0.0 ? d : e * d) * inv_rating, F);
  if (F == 0.0) grad = 0.0;
  return s * s;
}

template <int T, typename VT, bool RED>
__global__ void __launch_bounds__(NTHREADS, RED ? 3 : FDPF_MIN_BLOCKS)
    adjoint_tiles_kernel(FdpfParams P, AdjParams A, DevMatT<VT> M) {
  static_assert(T == 2 && Geo<T>::LP == 2, "one thread per row, two lanes: the slot sums need no atomics");
  __shared__ LaneState<T> L;
  __shared__ double red[NTHREADS * 2];  // lane_reduce and the loss sum
  RedLanes<T>* RL = nullptr;
  if constexpr (RED) {
    __shared__ RedLanes<T> rl;
    RL = &rl;
  }
  const Geo<T> g;
  const int tid = threadIdx.x;
  const DevGrid& G = P.G;
  VT* x = (VT*)P.wx + (size_t)blockIdx.x * P.vstride;
  VT* r = (VT*)P.wr + (size_t)blockIdx.x * P.vstride;
  VT* p = (VT*)P.wp + (size_t)blockIdx.x * P.vstride;
  VT* q = (VT*)P.wq + (size_t)blockIdx.x * P.vstride;
  VT* z = (VT*)P.wz + (size_t)blockIdx.x * P.vstride;
  const size_t so = (size_t)blockIdx.x * P.sstride;
  double* th = P.wth + so;   // theta by bus
  double* lm = P.wV + so;    // lambda by bus
  double* gP = A.gP + (size_t)blockIdx.x * G.n;
  double* gb = A.gb + (size_t)blockIdx.x * G.m;
  double* gf = A.g + (size_t)blockIdx.x * G.m * T;
  const int l0 = g.lane, l1 = g.lane + 1;
  for (int i = tid; i < G.n; i += NTHREADS) gP[i] = 0.0;
  for (int k = tid; k < G.m; k += NTHREADS) gb[k] = 0.0;
  double loss_acc = 0.0;
  __syncthreads();
  // tiles are dealt to CTAs statically (every scenario costs two solves), so
  // the per-slot sums, and hence the gradients, do not depend on timing
  for (int tile = blockIdx.x; tile < P.n_tiles; tile += gridDim.x) {
    if (tid < T) {
      const int ln = tid, s = tile * T + ln;
      const bool valid = s < P.S;
      const int l = valid ? P.sc.outage[s] : -1;
      L.scen[ln] = valid ? s : -1;
      L.l[ln] = l;
      L.lo[ln] = valid ? P.sc.isl_lo[s] : 0;
      L.cnt[ln] = valid ? P.sc.isl_cnt[s] : 0;
      L.coef[ln] = valid ? P.sc.coef[s] : 0.0;
      L.nogen[ln] = valid ? P.sc.no_gen[s] : 0;
      L.raP[ln] = l >= 0 ? M.row_of_bus[G.f[l]] : -1;
      L.rbP[ln] = l >= 0 ? M.row_of_bus[G.t[l]] : -1;
      L.wP[ln] = l >= 0 ? A.b[l] : 0.0;
      L.active[ln] = valid;
      L.inP[ln] = 0;
    }
    __syncthreads();
    const int lo0 = L.lo[l0], cnt0 = L.cnt[l0], lo1 = L.lo[l1], cnt1 = L.cnt[l1];
    const int br0 = L.l[l0], br1 = L.l[l1];
    const bool v0 = L.scen[l0] >= 0, v1 = L.scen[l1] >= 0;
    auto solve = [&]() {
      if constexpr (RED) red_solve<T, NTHREADS, VT>(P, M, L, *RL, r, L.raP, L.rbP, L.inP, nullptr);
      else pcg_solve<T, VT>(P, M, L, x, r, p, q, z, L.raP, L.rbP, L.wP, L.inP);
    };
    // the solution at matrix row k (-1: the slack)
    auto solution = [&](int k) {
      Pair<double> s{0.0, 0.0};
      if (k >= 0) {
        const Pair<VT> v = ld2((RED ? r : x) + (size_t)k * T + l0);
        s = {(double)v.a, (double)v.b};
        if constexpr (RED) s = {s.a * RL->xa[l0], s.b * RL->xa[l1]};
      }
      return s;
    };
    // right-hand side R_s P on the main island's non-slack rows
    for (int k = g.rs; k < M.n; k += Geo<T>::RPS) {
      const int i = M.bus_of_row[k], pr = M.pre_of_row[k];
      double pi = A.P[i];
      const double pg = G.bus_type[i] == 1 ? fmax(G.P_gen[i], 0.0) : 0.0;
      const double a = (v0 && !in_island(pr, lo0, cnt0)) ? pi + L.coef[l0] * pg : 0.0;
      const double b = (v1 && !in_island(pr, lo1, cnt1)) ? pi + L.coef[l1] * pg : 0.0;
      r[(size_t)k * T + g.lane] = (VT)a;
      r[(size_t)k * T + g.lane + 1] = (VT)b;
    }
    __syncthreads();
    solve();
    for (int i = g.rs; i < G.n; i += Geo<T>::RPS)
      st2(th + (size_t)i * T + g.lane, solution(M.row_of_bus[i]));
    __syncthreads();
    // loss over branches and g = dL/df, then y = A^T diag(b_s) g on the rows
    for (int k = g.rs; k < G.m; k += Geo<T>::RPS) {
      const int a = G.f[k], b = G.t[k];
      const int pa = G.pre[a], pb = G.pre[b];
      const double bk = A.b[k], ir = G.inv_rating[k];
      const Pair<double> ta = ld2(th + (size_t)a * T + l0), tb = ld2(th + (size_t)b * T + l0);
      Pair<double> gk{0.0, 0.0};
      if (v0 && k != br0 && !in_island(pa, lo0, cnt0) && !in_island(pb, lo0, cnt0))
        loss_acc += penalty(bk * (ta.a - tb.a), ir, gk.a);
      if (v1 && k != br1 && !in_island(pa, lo1, cnt1) && !in_island(pb, lo1, cnt1))
        loss_acc += penalty(bk * (ta.b - tb.b), ir, gk.b);
      st2(gf + (size_t)k * T + l0, gk);
    }
    __syncthreads();
    for (int k = g.rs; k < M.n; k += Geo<T>::RPS) {
      const int i = M.bus_of_row[k], pr = M.pre_of_row[k];
      const bool m0 = v0 && !in_island(pr, lo0, cnt0), m1 = v1 && !in_island(pr, lo1, cnt1);
      double y0 = 0.0, y1 = 0.0;
      for (int e = G.adj_ptr[i]; e < G.adj_ptr[i + 1]; ++e) {
        const int br = G.adj_br[e];
        const double bk = G.f[br] == i ? A.b[br] : -A.b[br];
        const Pair<double> gk = ld2(gf + (size_t)br * T + l0);
        if (m0) y0 = fma(bk, gk.a, y0);
        if (m1) y1 = fma(bk, gk.b, y1);
      }
      r[(size_t)k * T + g.lane] = (VT)y0;
      r[(size_t)k * T + g.lane + 1] = (VT)y1;
    }
    __syncthreads();
    solve();
    // lambda by bus; the re-dispatch transpose needs sum_k P_gen,k lambda_k
    // and sum_k P_gen,k over the main island's PV buses
    double wl0 = 0.0, wl1 = 0.0, dn0 = 0.0, dn1 = 0.0;
    for (int i = g.rs; i < G.n; i += Geo<T>::RPS) {
      const Pair<double> l = solution(M.row_of_bus[i]);
      const double a = l.a, b = l.b;
      st2(lm + (size_t)i * T + g.lane, l);
      if (G.bus_type[i] == 1 && G.P_gen[i] > 0.0) {
        const int pr = G.pre[i];
        const double pg = G.P_gen[i];
        if (!in_island(pr, lo0, cnt0)) { wl0 += pg * a; dn0 += pg; }
        if (!in_island(pr, lo1, cnt1)) { wl1 += pg * b; dn1 += pg; }
      }
    }
    const Pair<double> WL = lane_reduce<T, false>(red, wl0, wl1);
    const Pair<double> DN = lane_reduce<T, false>(red, dn0, dn1);
    const double W0 = (v0 && cnt0 > 0 && !L.nogen[l0] && DN.a > 0.0) ? WL.a / DN.a : 0.0;
    const double W1 = (v1 && cnt1 > 0 && !L.nogen[l1] && DN.b > 0.0) ? WL.b / DN.b : 0.0;
    for (int i = g.rs; i < G.n; i += Geo<T>::RPS) {
      const int pr = G.pre[i];
      double add = 0.0;
      if (v0) add += in_island(pr, lo0, cnt0) ? W0 : lm[(size_t)i * T + l0];
      if (v1) add += in_island(pr, lo1, cnt1) ? W1 : lm[(size_t)i * T + l1];
      gP[i] += add;
    }
    for (int k = g.rs; k < G.m; k += Geo<T>::RPS) {
      const int a = G.f[k], b = G.t[k];
      const int pa = G.pre[a], pb = G.pre[b];
      const Pair<double> gk = ld2(gf + (size_t)k * T + l0);
      const Pair<double> ta = ld2(th + (size_t)a * T + l0), tb = ld2(th + (size_t)b * T + l0);
      const Pair<double> la = ld2(lm + (size_t)a * T + l0), lb = ld2(lm + (size_t)b * T + l0);
      double add = 0.0;
      if (v0 && k != br0 && !in_island(pa, lo0, cnt0) && !in_island(pb, lo0, cnt0))
        add = (ta.a - tb.a) * (gk.a - (la.a - lb.a));
      if (v1 && k != br1 && !in_island(pa, lo1, cnt1) && !in_island(pb, lo1, cnt1))
        add = fma(ta.b - tb.b, gk.b - (la.b - lb.b), add);
      gb[k] += add;
    }
    __syncthreads();
  }
  // the CTA's loss: sum over threads in a fixed order
  red[tid] = loss_acc;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int k = 0; k < NTHREADS; ++k) s += red[k];
    A.loss[blockIdx.x] = s;
  }
}

// out[map[i]] = sum over slots of acc[slot][i], in a fixed order: 16 threads
// per element take every 16th slot, then a tree over them.
constexpr int SUM_COLS = 32, SUM_ROWS = 16;
__global__ void __launch_bounds__(SUM_COLS* SUM_ROWS)
    slot_sum_kernel(int n, int slots, const double* __restrict__ acc,
                    const int32_t* __restrict__ map, double* out) {
  __shared__ double part[SUM_ROWS][SUM_COLS + 1];
  const int i = blockIdx.x * SUM_COLS + threadIdx.x;
  double s = 0.0;
  if (i < n)
    for (int k = threadIdx.y; k < slots; k += SUM_ROWS) s += acc[(size_t)k * n + i];
  part[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  for (int h = SUM_ROWS / 2; h > 0; h >>= 1) {
    if (threadIdx.y < h) part[threadIdx.y][threadIdx.x] += part[threadIdx.y + h][threadIdx.x];
    __syncthreads();
  }
  if (i < n && threadIdx.y == 0) out[map ? map[i] : i] = part[0][threadIdx.x];
}

__global__ void gather_perm_kernel(int n, const int32_t* __restrict__ idx,
                                   const double* __restrict__ src, double* dst) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[idx[i]];
}

cudaError_t launch_adjoint(cudaStream_t st, int grid, const FdpfParams& P, const AdjParamsView& A,
                           const DevMatT<double>& M) {
  AdjParams a;
  a.P = A.P;
  a.b = A.b;
  a.gP = A.gP;
  a.gb = A.gb;
  a.loss = A.loss;
  a.g = A.g;
  if (reduced_form(P.precond, M, M))
    adjoint_tiles_kernel<2, double, true><<<grid, NTHREADS, 0, st>>>(P, a, M);
  else
    adjoint_tiles_kernel<2, double, false><<<grid, NTHREADS, 0, st>>>(P, a, M);
  return cudaGetLastError();
}

int adjoint_max_blocks_per_sm(bool red) {
  int nb = 0;
  if (red)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, adjoint_tiles_kernel<2, double, true>,
                                                  NTHREADS, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, adjoint_tiles_kernel<2, double, false>,
                                                  NTHREADS, 0);
  return nb;
}

cudaError_t launch_slot_sum(cudaStream_t st, int n, int slots, const double* acc,
                            const int32_t* map, double* out) {
  if (n > 0)
    slot_sum_kernel<<<(n + SUM_COLS - 1) / SUM_COLS, dim3(SUM_COLS, SUM_ROWS), 0, st>>>(
        n, slots, acc, map, out);
  return cudaGetLastError();
}

cudaError_t launch_gather_perm(cudaStream_t st, int n, const int32_t* idx, const double* src,
                               double* dst) {
  if (n > 0) gather_perm_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, idx, src, dst);
  return cudaGetLastError();
}

}  // namespace gpcg
