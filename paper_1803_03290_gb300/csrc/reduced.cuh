// The base-preconditioned CG of one outage in its two-dimensional Krylov
// space, for the complete base-case factor.
//
// With M = B = L L^T the base-case matrix itself and B_s = B - w v v^T the
// outage's (v = c e_from - e_to), M^-1 B_s maps span{z0, y}, z0 = M^-1 r0 and
// y = M^-1 v_m, into itself: B_s z = B z - w (v.z) v_m on the main island
// (v_m: v without an islanded end, which is masked out of every vector).  So
// every iterate of the PCG of Sec. IV.B is a combination of those two
// vectors and every residual one of r0 and v_m, and the recurrence needs
// only scalars:
//   r.r    from r0.r0, v_m.r0, v_m.v_m,
//   r.z    from r0.z0 = |L^-1 r0|^2, v_m.z0 and v_m.y,
//   v.z    from v.z0 = (L^-1 v).(L^-1 r0) and v.y.
// All of them are known after the forward substitution f = L^-1 r0: L^-1 v
// and L^-1 v_m are sparse (the ancestors of the outage's ends in the
// elimination tree, about 60 of 10,000 rows) and belong to the grid
// (BranchCols).  The solution xa z0 + xb y = xa L^-T (f + (xb / xa) L^-1 v_m)
// then takes one backward substitution.  An inner solve is one forward and one
// backward pass over one vector in place of an SpMV, a forward and a backward
// pass over five vectors per iteration, with the same iterates and the same
// stopping rule.  10,000 buses, all 13,500 outages, 1e-4 p.u.: with FP64 vectors
// every iteration count is that of the five-vector PCG, with FP32 vectors they
// are those counts too (3.81 P iterations a scenario; the five-vector PCG's FP32
// residuals asked for 3.88).  Screen 163 -> 102 ms with FP64 vectors; 3,001 outages
// at 1e-10 p.u. with FP32 ones 62.9 -> 41.0 ms.  reduced_form (fdpf.h) says which
// screens take it.
#pragma once
#include "fdpf_ops.cuh"

namespace gpcg {

// The dense products of the tail: the threads are split into as many groups as
// the tail's rows (rounded up to warps) fit the CTA's row slots, a group takes
// every groups-th term of each row, and the first one adds the shares up.  TR: X^T
// (row-major xr, terms from the diagonal of the warp's first row) or X (column-
// major xc, terms up to the diagonal of the warp's last row); either way
// consecutive threads read consecutive values.
template <int T, int NT, int NL, bool TR, typename VT>
__device__ __forceinline__ bool tail_product(const VT* __restrict__ X, int nt,
                                             const VT* __restrict__ s, VT* __restrict__ part,
                                             int& k, Vec<VT, Geo<T, NT>::LP>& a) {
  constexpr int LP = Geo<T, NT>::LP, RPS = Geo<T, NT>::RPS, UN = NT == 1024 ? 16 : 8;
  const Geo<T, NT> g;
  a = vzero<VT, LP>();
  if constexpr (RPS >= 32 && Geo<T, NT>::TPR == 1) {
    const int pad = (nt + 31) & ~31, ng = RPS / pad;  // ng >= 1: nt <= 248 < RPS
    const int q = g.rs / pad;
    k = g.rs - q * pad;
    if (q < ng) {  // whole warps
      const int first = TR ? (k & ~31) + q : q;
      const int last = TR ? nt : min(nt, (k | 31) + 1);
      if (k < nt) {
        const VT* col = X + k;
#pragma unroll UN
        for (int j = first; j < last; j += ng) {
          const VT xv = __ldg(col + (size_t)j * nt);
          const Vec<VT, LP> sv = ldv<LP>(s + (size_t)j * T + g.lane);
#pragma unroll
          for (int l = 0; l < NL; ++l) a.v[l] += xv * sv.v[l];
        }
        if (q) stv<LP>(part + ((size_t)(q - 1) * pad + k) * T + g.lane, a);
      }
    }
    __syncthreads();
    if (q || k >= nt) return false;
    for (int h = 0; h < ng - 1; ++h) {
      const Vec<VT, LP> u = ldv<LP>(part + ((size_t)h * pad + k) * T + g.lane);
#pragma unroll
      for (int l = 0; l < NL; ++l) a.v[l] += u.v[l];
    }
    return true;
  }
  return false;
}
// Shared memory of the groups' shares.
template <int T, int NT>
constexpr int TAIL_PART = Geo<T, NT>::TPR == 1 ? Geo<T, NT>::RPS * T : 1;

// One row of a substitution as its table holds it.
template <typename VT>
struct SubRow {
  int4 rc;
  int4 c;
  VT v[SUB_K], id;
};
template <typename VT>
__device__ __forceinline__ SubRow<VT> sub_row(const SubTab<VT>& tab, int e) {
  SubRow<VT> r;
  r.rc = __ldg(tab.rc + e);
  r.c = __ldg(tab.col + e);
  ld_vals<SUB_K>(tab.val + (size_t)e * SUB_K, r.v);
  r.id = __ldg(tab.id + e);
  return r;
}
// a - (the row's entries times the solved values), times 1 / L_ii; the first NL
// lanes of the thread.
template <int T, int NL, typename VT, int LP>
__device__ __forceinline__ void sub_apply(const SubRow<VT>& w, const SubTab<VT>& tab,
                                          const VT* __restrict__ f, int lane, Vec<VT, LP>& a) {
  const int c[SUB_K] = {w.c.x, w.c.y, w.c.z, w.c.w};
#pragma unroll
  for (int k = 0; k < SUB_K; ++k)
    if (k < w.rc.y) {
      const Vec<VT, LP> z = ldv<LP>(f + (size_t)c[k] * T + lane);
#pragma unroll
      for (int j = 0; j < NL; ++j) a.v[j] -= w.v[k] * z.v[j];
    }
  for (int h = w.rc.z, left = w.rc.y - SUB_K; left > 0; ++h, left -= SUB_K) {
    const int4 cc = __ldg(tab.ccol + h);
    const int d[SUB_K] = {cc.x, cc.y, cc.z, cc.w};
    VT v[SUB_K];
    ld_vals<SUB_K>(tab.cval + (size_t)h * SUB_K, v);
#pragma unroll
    for (int k = 0; k < SUB_K; ++k)
      if (k < left) {
        const Vec<VT, LP> z = ldv<LP>(f + (size_t)d[k] * T + lane);
#pragma unroll
        for (int j = 0; j < NL; ++j) a.v[j] -= v[k] * z.v[j];
      }
  }
#pragma unroll
  for (int j = 0; j < NL; ++j) a.v[j] *= w.id;
}
// Whether a row is loaded a level ahead of its use: in the wide CTAs, whose
// levels are a row or less per thread and wait on nothing else.
template <int NT>
constexpr bool SUB_AHEAD = NT > NTHREADS;

// Forward substitution f = L^-1 r in place over the levels before the tail,
// and the tail's right-hand side reduced and multiplied by the tail's dense
// inverse (y into zt).  Adds the lanes' partial |r|^2 to rr and |f|^2 to ff.
// NL: the thread's lanes that hold a scenario (FP64 solves of a tile with one).
template <int T, int NT, int NL, typename VT>
__device__ __forceinline__ void red_forward(const DevMatT<VT>& M, VT* __restrict__ f,
                                            VT* __restrict__ zt, VT* __restrict__ part,
                                            Vec<VT, Geo<T, NT>::LP>& rr,
                                            Vec<VT, Geo<T, NT>::LP>& ff) {
  constexpr int LP = Geo<T, NT>::LP;
  const Geo<T, NT> g;
  constexpr int RPS = Geo<T, NT>::RPS, NPT = (TAIL_ROWS + RPS - 1) / RPS;
  const int nl = M.tail_lev, t0 = M.tail_row0, nt = M.n - t0;
  int r0 = 0, r1 = nl > 0 ? __ldg(M.lev_ptr + 1) : 0;
  SubRow<VT> nx;
  int at = -1;
  if (SUB_AHEAD<NT> && g.rs < r1) nx = sub_row(M.fwd, at = g.rs);
  for (int lev = 0; lev < nl; ++lev) {
    const int r2 = lev + 1 < nl ? __ldg(M.lev_ptr + lev + 2) : r1;
    for (int e = r0 + g.rs; e < r1; e += RPS) {
      SubRow<VT> w;
      if (SUB_AHEAD<NT> && at == e) w = nx;
      else w = sub_row(M.fwd, e);
      if (SUB_AHEAD<NT>) {
        const int ne = e + RPS < r1 ? e + RPS : r1 + g.rs < r2 ? r1 + g.rs : -1;
        if (ne >= 0) nx = sub_row(M.fwd, at = ne);
      }
      const size_t o = (size_t)w.rc.x * T + g.lane;
      Vec<VT, LP> a = ldv<LP>(f + o);
#pragma unroll
      for (int j = 0; j < NL; ++j) rr.v[j] += a.v[j] * a.v[j];
      sub_apply<T, NL>(w, M.fwd, f, g.lane, a);
#pragma unroll
      for (int j = 0; j < NL; ++j) ff.v[j] += a.v[j] * a.v[j];
      stv<LP>(f + o, a);
    }
    // a thread without a row in this level: its row of the next one
    if (SUB_AHEAD<NT> && at < r1 && r1 + g.rs < r2) nx = sub_row(M.fwd, at = r1 + g.rs);
    __syncthreads();
    r0 = r1;
    r1 = r2;
  }
  if (nt <= 0) return;
  // the tail rows' right-hand side, minus the rows solved before: TH threads per
  // row (the rows have up to dozens of such entries, each a chain of two loads)
  constexpr int TPR = Geo<T, NT>::TPR, TH = TPR >= 32 ? 1 : 32 / TPR < 8 ? 32 / TPR : 8;
  const int h = g.rs % TH;
  for (int k0 = 0; k0 < nt; k0 += RPS / TH) {  // every thread takes part in the sums
    const int k = k0 + g.rs / TH;
    Vec<VT, LP> a = vzero<VT, LP>();
    if (k < nt) {
      const int e1 = __ldg(M.th_ptr + k + 1);
      for (int e = __ldg(M.th_ptr + k) + h; e < e1; e += TH) {
        const VT vv = __ldg(M.th_val + e);
        const Vec<VT, LP> zz = ldv<LP>(f + (size_t)__ldg(M.th_col + e) * T + g.lane);
#pragma unroll
        for (int j = 0; j < NL; ++j) a.v[j] += vv * zz.v[j];
      }
    }
#pragma unroll
    for (int off = TH / 2; off > 0; off >>= 1)
#pragma unroll
      for (int j = 0; j < NL; ++j) a.v[j] += __shfl_xor_sync(0xffffffffu, a.v[j], off * TPR);
    if (k < nt && h == 0) {
      Vec<VT, LP> r = ldv<LP>(f + (size_t)(t0 + k) * T + g.lane);
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        rr.v[j] += r.v[j] * r.v[j];
        r.v[j] -= a.v[j];
      }
      stv<LP>(zt + (size_t)k * T + g.lane, r);
    }
  }
  __syncthreads();
  // y_t = X rhs: X_kj = xc[j nt + k], zero above the diagonal
  if constexpr (TPR == 1) {
    int k;
    Vec<VT, LP> y;
    if (tail_product<T, NT, NL, false>(M.xc, nt, zt, part, k, y)) {
#pragma unroll
      for (int l = 0; l < NL; ++l) ff.v[l] += y.v[l] * y.v[l];
      stv<LP>(zt + (size_t)k * T + g.lane, y);
    }
  } else {
    Vec<VT, LP> y[NPT];
#pragma unroll
    for (int m = 0; m < NPT; ++m) {
      const int k = g.rs + m * RPS;
      const int jend = min(nt, __shfl_sync(0xffffffffu, k, 31) + 1);  // every lane takes part
      y[m] = vzero<VT, LP>();
      if (k < nt) {
        const VT* col = M.xc + k;
#pragma unroll 4
        for (int j = 0; j < jend; ++j) {
          const VT xv = __ldg(col + (size_t)j * nt);
          const Vec<VT, LP> sv = ldv<LP>(zt + (size_t)j * T + g.lane);
#pragma unroll
          for (int l = 0; l < NL; ++l) y[m].v[l] += xv * sv.v[l];
        }
#pragma unroll
        for (int l = 0; l < NL; ++l) ff.v[l] += y[m].v[l] * y[m].v[l];
      }
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < NPT; ++m) {
      const int k = g.rs + m * RPS;
      if (k < nt) stv<LP>(zt + (size_t)k * T + g.lane, y[m]);
    }
  }
}

// Backward substitution x = L^-T f in place, the tail first (its y in zt).
template <int T, int NT, int NL, typename VT>
__device__ __forceinline__ void red_backward(const DevMatT<VT>& M, VT* __restrict__ f,
                                             const VT* __restrict__ zt,
                                             VT* __restrict__ part) {
  constexpr int LP = Geo<T, NT>::LP;
  const Geo<T, NT> g;
  constexpr int RPS = Geo<T, NT>::RPS, NPT = (TAIL_ROWS + RPS - 1) / RPS;
  const int t0 = M.tail_row0, nt = M.n - t0;
  if (nt > 0) {
    // z_t = X^T y_t: X_ik = xr[i nt + k], zero for i < k
    if constexpr (Geo<T, NT>::TPR == 1) {
      int k;
      Vec<VT, LP> a;
      if (tail_product<T, NT, NL, true>(M.xr, nt, zt, part, k, a))
        stv<LP>(f + (size_t)(t0 + k) * T + g.lane, a);
    } else {
#pragma unroll
      for (int m = 0; m < NPT; ++m) {
        const int k = g.rs + m * RPS;
        const int ibeg = __shfl_sync(0xffffffffu, k, 0);
        if (k >= nt) continue;
        const VT* col = M.xr + k;
        Vec<VT, LP> a = vzero<VT, LP>();
#pragma unroll 4
        for (int i = ibeg; i < nt; ++i) {
          const VT xv = __ldg(col + (size_t)i * nt);
          const Vec<VT, LP> sv = ldv<LP>(zt + (size_t)i * T + g.lane);
#pragma unroll
          for (int l = 0; l < NL; ++l) a.v[l] += xv * sv.v[l];
        }
        stv<LP>(f + (size_t)(t0 + k) * T + g.lane, a);
      }
    }
    __syncthreads();
  }
  const int nb = M.ntblev;
  int r0 = nb > 0 ? __ldg(M.tblev_ptr) : 0, r1 = nb > 0 ? __ldg(M.tblev_ptr + 1) : 0;
  SubRow<VT> nx;
  int at = -1;
  if (SUB_AHEAD<NT> && r0 + g.rs < r1) nx = sub_row(M.bwd, at = r0 + g.rs);
  for (int lev = 0; lev < nb; ++lev) {
    const int r2 = lev + 1 < nb ? __ldg(M.tblev_ptr + lev + 2) : r1;
    for (int e = r0 + g.rs; e < r1; e += RPS) {
      SubRow<VT> w;
      if (SUB_AHEAD<NT> && at == e) w = nx;
      else w = sub_row(M.bwd, e);
      if (SUB_AHEAD<NT>) {
        const int ne = e + RPS < r1 ? e + RPS : r1 + g.rs < r2 ? r1 + g.rs : -1;
        if (ne >= 0) nx = sub_row(M.bwd, at = ne);
      }
      const size_t o = (size_t)w.rc.x * T + g.lane;
      Vec<VT, LP> a = ldv<LP>(f + o);
      sub_apply<T, NL>(w, M.bwd, f, g.lane, a);
      stv<LP>(f + o, a);
    }
    if (SUB_AHEAD<NT> && at < r1 && r1 + g.rs < r2) nx = sub_row(M.bwd, at = r1 + g.rs);
    __syncthreads();
    r0 = r1;
    r1 = r2;
  }
}

// What a lane's recurrence starts from: R = r0.r0, Z = r0.z0, u = v.z0,
// m0 = v_m.z0, vr = v_m.r0, and the branch's scalars.
struct RedScalars {
  double R, Z, u, m0, vr, vy, my, vm2, w;
};

// The PCG of pcg_solve on those scalars: same steps, same stopping rule.
// The solution is xa z0 + xb y; returns the iterations taken.
__device__ inline int reduced_cg(const RedScalars& q, double tol2, int max_inner, double& xa,
                                 double& xb) {
  xa = xb = 0.0;
  if (!(q.R > 0.0) || !(q.Z > 0.0)) return 0;
  double a = 1.0, b = 0.0, pa = 1.0, pb = 0.0, rz = q.Z, best = q.R;
  int its = 0, stall = 0;
  while (its < max_inner) {
    const double qb = pb - q.w * (pa * q.u + pb * q.vy);  // B_s p = pa r0 + qb v_m
    const double pq = pa * pa * q.Z + (pa * qb + pb * pa) * q.m0 + pb * qb * q.my;
    if (!(pq > 0.0) || !isfinite(pq)) break;
    const double al = rz / pq;
    xa += al * pa;
    xb += al * pb;
    a -= al * pa;
    b -= al * qb;
    ++its;
    const double rr = a * a * q.R + 2.0 * a * b * q.vr + b * b * q.vm2;
    if (!(rr > tol2 * q.R) || !isfinite(rr)) break;
    if (rr < 0.999 * best) { best = rr; stall = 0; }
    else if (++stall >= STALL_ITERS) break;
    if (rr > 1e4 * best) break;
    const double rzn = a * a * q.Z + 2.0 * a * b * q.m0 + b * b * q.my;
    if (!(rzn > 0.0)) break;
    const double be = rzn / rz;
    rz = rzn;
    pa = a + be * pa;
    pb = b + be * pb;
  }
  return its;
}

// ------------------------------------------------- with extension rows
// A lane with nx extension rows (B'' rows of switched buses) solves
//   [ B_s  C ; C^T  D ],  C's columns the couplings c_s, preconditioned by
//   [ M ; diag D ].
// The matrix rows' part of every vector then lies in the span of 2 + nx known
// ones, r0, v_m and the c_s (their M^-1 images for iterates), and the extension
// rows are coordinates of their own, so the PCG of pcg_solve runs on at most 10
// + 8 coordinates with
//   G_ij = rho_i.M^-1 rho_j = f_i.f_j,  N_ij = rho_i.rho_j,  u_i = v.M^-1 rho_i.
// The f_s = L^-1 c_s are sparse (BusCols; about 20 rows per bus, the PV buses cut
// B'' into small pieces).  If the outaged branch joins a switched bus to row o,
// its coupling is not part of c_s: c_s = c_b + k v, as v has only the entry at o.
// Measured: 1,999 generator outages of 10,000 buses at 1e-10 p.u. 76.6 -> 46.9 ms,
// 2,700 outages of 2,000 buses with reactive limits 38.9 -> 13.5 ms.
constexpr int RX = 2 + KX;  // coordinates on the matrix rows
template <int T>
struct RedExt {
  double G[T][RX][RX], N[T][RX][RX], u[T][RX];
  double D[T][KX][KX];
  double k[T][KX];   // c_s = c_b + k v
  double xe[T][KX];  // right-hand side, then solution on the extension rows
};

// Couplings of extension row s of lane ln without the outaged branch: visit(row,
// value) per matrix row, and the branch's own value at row o (bo), if any.
template <typename VT, typename F>
__device__ __forceinline__ void ext_couplings(const DevMatT<VT>& M, int b, int lb, F visit) {
  const int e1 = __ldg(M.xptr + b + 1);
  for (int e = __ldg(M.xptr + b); e < e1; ++e) {
    const int rw = __ldg(M.xrow + e);
    if (rw >= 0 && __ldg(M.xbr + e) != lb) visit(rw, (double)__ldg(M.xval + e));
  }
}

// What has to be taken from r0 before the forward pass overwrites it: N_0j, the
// right-hand side on the extension rows, D and the c_s dot products; thread
// `ln`, one per lane.
template <int T, int NT, typename VT>
__device__ __noinline__ void ext_setup(const DevMatT<VT>& M, const LaneState<T, NT>& L,
                                       const SwitchState<T>& SW, RedExt<T>& X, const VT* f,
                                       int ln, int ra, int rb, double w, double c) {
  const int nx = SW.nx[ln], l = L.l[ln];
  double ca = 0.0, cb = 0.0;
  if (l >= 0) {
    const double* sc = M.br.sc + (size_t)l * SC_N;
    ca = sc[SC_CA];
    cb = sc[SC_CB];
  }
  for (int s = 0; s < nx; ++s) {
    const int b = SW.xb[ln][s];
    X.xe[ln][s] = (double)f[(size_t)(M.n + 1 + s) * T + ln];
    // v = c e_ra - e_rb has the other end's entry only when b is an end
    X.k[ln][s] = b == L.fb[ln] ? (rb >= 0 ? -w * c : 0.0) : b == L.tb[ln] ? (ra >= 0 ? w : 0.0) : 0.0;
    double r0 = 0.0, vm = 0.0;
    ext_couplings(M, b, l, [&](int rw, double v) {
      r0 = fma(v, (double)f[(size_t)rw * T + ln], r0);
      if (rw == ra) vm = fma(v, ca, vm);
      if (rw == rb) vm = fma(v, cb, vm);
    });
    X.N[ln][0][2 + s] = X.N[ln][2 + s][0] = r0;
    X.N[ln][1][2 + s] = X.N[ln][2 + s][1] = vm;
    for (int t = 0; t <= s; ++t) {
      double cc = 0.0, d = 0.0;
      const int bt = SW.xb[ln][t];
      ext_couplings(M, b, l, [&](int rw, double v) {
        ext_couplings(M, bt, l, [&](int rt, double vt) {
          if (rt == rw) cc = fma(v, vt, cc);
        });
      });
      if (t == s) {
        // the diagonal without the outaged branch's term
        d = (double)M.xdiag[b];
        if (b == L.fb[ln]) d -= w * c * c;
        else if (b == L.tb[ln]) d -= w;
      } else {
        const int e1 = __ldg(M.xptr + b + 1);
        for (int e = __ldg(M.xptr + b); e < e1; ++e)
          if (__ldg(M.xnb + e) == bt && __ldg(M.xbr + e) != l) d += (double)__ldg(M.xval + e);
      }
      X.N[ln][2 + s][2 + t] = X.N[ln][2 + t][2 + s] = cc;
      X.D[ln][s][t] = X.D[ln][t][s] = d;
    }
  }
}

// Position of row i in the sorted rows [e0, e1), or -1.
__device__ __forceinline__ int find_row(const int32_t* __restrict__ row, int e0, int e1, int i) {
  while (e0 < e1) {
    const int mid = (e0 + e1) >> 1, r = __ldg(row + mid);
    if (r == i) return mid;
    if (r < i) e0 = mid + 1; else e1 = mid;
  }
  return -1;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// The lane's coordinates and the PCG on them, by one warp (all 32 threads): thread
// i < 2 + nx holds coordinate i, thread 16 + s the extension row s.  q: the scalars
// of r0 and v as reduced_cg takes them.  Returns the iterations; on return x is
// the thread's coordinate of the solution.
template <int T, int NT, typename VT, typename AT>
__device__ __noinline__ int ext_solve(const DevMatT<VT>& M, const LaneState<T, NT>& L,
                                      const SwitchState<T>& SW, RedExt<T>& X,
                                      const RedScalars& q, int ln, AT at, double tol2,
                                      int max_inner, double& x) {
  const int wl = threadIdx.x & 31, nx = SW.nx[ln], K = 2 + nx, l = L.l[ln];
  auto& G = X.G[ln];
  auto& N = X.N[ln];
  double vv = 0.0;
  int e0 = 0, e1 = 0;
  if (l >= 0) {
    vv = __ldg(M.br.sc + (size_t)l * SC_N + SC_VV);
    e0 = __ldg(M.br.ptr + l);
    e1 = __ldg(M.br.ptr + l + 1);
  }
  if (wl == 0) {
    G[0][0] = q.Z; G[0][1] = G[1][0] = q.m0; G[1][1] = q.my;
    N[0][0] = q.R; N[0][1] = N[1][0] = q.vr; N[1][1] = q.vm2;
    X.u[ln][0] = q.u;
    X.u[ln][1] = q.vy;
  }
  for (int s = 0; s < nx; ++s) {
    const int b = SW.xb[ln][s], s0 = __ldg(M.bus.ptr + b), s1 = __ldg(M.bus.ptr + b + 1);
    const double ks = X.k[ln][s];
    double h = 0.0, a = 0.0, m = 0.0;  // f_b with f0, L^-1 v, L^-1 v_m
    for (int e = s0 + wl; e < s1; e += 32) {
      const int i = __ldg(M.bus.row + e);
      const double fb = __ldg(M.bus.f + e);
      h = fma(fb, (double)*at(i), h);
      if (l >= 0) {
        const int p = find_row(M.br.row, e0, e1, i);
        if (p >= 0) {
          a = fma(fb, __ldg(M.br.fv + p), a);
          m = fma(fb, __ldg(M.br.fm + p), m);
        }
      }
    }
    h = warp_sum(h);
    a = warp_sum(a);
    m = warp_sum(m);
    if (wl == 0) {
      G[0][2 + s] = G[2 + s][0] = fma(ks, q.u, h);
      G[1][2 + s] = G[2 + s][1] = fma(ks, q.vy, m);
      X.u[ln][2 + s] = fma(ks, vv, a);
      G[2 + s][2 + s] = __ldg(M.bus.ff + b) + ks * (2.0 * a + ks * vv);
    }
    for (int t = 0; t < s; ++t) {
      const int bt = SW.xb[ln][t], t0 = __ldg(M.bus.ptr + bt), t1 = __ldg(M.bus.ptr + bt + 1);
      double d = 0.0;
      for (int e = s0 + wl; e < s1; e += 32) {
        const int p = find_row(M.bus.row, t0, t1, __ldg(M.bus.row + e));
        if (p >= 0) d = fma(__ldg(M.bus.f + e), __ldg(M.bus.f + p), d);
      }
      d = warp_sum(d);
      __syncwarp();
      if (wl == 0) {
        // f_s.f_t with f_s = f_b + ks fv: u holds v.M^-1 c_t with its own kt
        const double kt = X.k[ln][t], at_ = X.u[ln][2 + t] - kt * vv;
        G[2 + s][2 + t] = G[2 + t][2 + s] = d + ks * at_ + kt * a + ks * kt * vv;
      }
    }
    __syncwarp();
  }
  __syncwarp();
  const bool mn = wl < K, ex = wl >= 16 && wl < 16 + nx;
  const int s = wl - 16;
  const double gd = ex ? X.D[ln][s][s] : 0.0;
  auto row_dot = [&](const double (&A)[RX][RX], double v) {  // (A v)_wl
    double r = 0.0;
    for (int j = 0; j < K; ++j) {
      const double vj = __shfl_sync(0xffffffffu, v, j);
      if (mn) r = fma(A[wl][j], vj, r);
    }
    return r;
  };
  double r = mn ? (wl == 0 ? 1.0 : 0.0) : ex ? X.xe[ln][s] : 0.0;
  x = 0.0;
  auto pre = [&](double v) { return ex ? (gd > 0.0 ? v / gd : 0.0) : v; };
  const double n0 = row_dot(N, r);  // (every thread takes part in the shuffles)
  const double bb = warp_sum(mn ? r * n0 : r * r);
  double z = pre(r);
  double gz = row_dot(G, z);
  double rz = warp_sum(mn ? r * gz : r * z);
  if (!(bb > 0.0) || !(rz > 0.0)) return 0;
  double p = z, best = bb;
  int its = 0, stall = 0;
  while (its < max_inner) {
    // q = B_ext p: main coordinates, and the extension rows
    const double gp = row_dot(G, p);
    double up = 0.0, qe = 0.0;
    for (int j = 0; j < K; ++j) {
      const double pj = __shfl_sync(0xffffffffu, p, j);
      up = fma(X.u[ln][j], pj, up);
      if (ex) qe = fma(G[2 + s][j], pj, qe);
    }
    for (int t = 0; t < nx; ++t) {
      const double pt = __shfl_sync(0xffffffffu, p, 16 + t);
      if (ex) qe = fma(X.D[ln][s][t], pt, qe);
    }
    const double pe = __shfl_sync(0xffffffffu, p, wl >= 2 && wl < K ? 14 + wl : 31);
    double qv = mn ? p : ex ? qe : 0.0;
    if (wl == 1) qv -= q.w * up;
    if (mn && wl >= 2) qv += pe;
    const double pq = warp_sum(mn ? qv * gp : ex ? p * qv : 0.0);
    if (!(pq > 0.0) || !isfinite(pq)) break;
    const double al = rz / pq;
    x = fma(al, p, x);
    r = fma(-al, qv, r);
    ++its;
    const double nr = row_dot(N, r);
    const double rr = warp_sum(mn ? r * nr : ex ? r * r : 0.0);
    if (!(rr > tol2 * bb) || !isfinite(rr)) break;
    if (rr < 0.999 * best) { best = rr; stall = 0; }
    else if (++stall >= STALL_ITERS) break;
    if (rr > 1e4 * best) break;
    z = pre(r);
    gz = row_dot(G, z);
    const double rzn = warp_sum(mn ? r * gz : ex ? r * z : 0.0);
    if (!(rzn > 0.0)) break;
    const double be = rzn / rz;
    rz = rzn;
    p = fma(be, p, z);
  }
  return its;
}

template <int T, int NT = NTHREADS>
struct RedLanes {
  double vr[T], xa[T];
  double part[2][NT / 32][T];  // the warps' partial r.r and |f|^2
};

// PCG on B_s x = f for the lanes that are active and not held, f in place:
// on return lane s's solution is S.xa[s] times the vector (xa = 0: no step).
// Adds each lane's iteration count to iters.
//
// EXT: lanes may have extension rows (SW, X; w, c: the lanes' branch weights and
// from-end factors); their solution is left in X.xe.
template <int T, int NT, typename VT, bool EXT = false>
__device__ GPCG_PASS_INLINE void red_solve(const FdpfParams& P, const DevMatT<VT>& M,
                                           LaneState<T, NT>& L, RedLanes<T, NT>& S, VT* f,
                                           const int* ra, const int* rb, int* iters,
                                           const int* hold, const SwitchState<T>* SW = nullptr,
                                           RedExt<T>* X = nullptr, const double* w = nullptr,
                                           const double* c = nullptr) {
  constexpr int LP = Geo<T, NT>::LP;
  constexpr int NW = NT / 32, TPR = Geo<T, NT>::TPR;
  __shared__ __align__(16) VT zt[TAIL_ROWS * T];
  __shared__ __align__(16) VT part[TAIL_PART<T, NT>];
  const Geo<T, NT> g;
  const int tid = threadIdx.x, warp = tid >> 5, wl = tid & 31;
  // diagnostics (P.phase_cycles set): thread 0's SM cycles between the barriers
  // (recurrence, forward, backward), in the slots after the per-scenario times
  const bool tim = P.phase_cycles != nullptr && tid == 0;
  long long tm = tim ? clock64() : 0;
  auto lap = [&](int k) {
    if (!tim) return;
    const long long t = clock64();
    atomicAdd(P.phase_cycles + 8 + 2 * (size_t)P.S + k, (unsigned long long)(t - tm));
    tm = t;
  };
  if (tid < T) {  // v_m.r0, before f is overwritten; the zero row of the padding
    double vr = 0.0;
    if (L.active[tid] && L.l[tid] >= 0) {
      const double* sc = M.br.sc + (size_t)L.l[tid] * SC_N;
      if (ra[tid] >= 0) vr += sc[SC_CA] * (double)f[(size_t)ra[tid] * T + tid];
      if (rb[tid] >= 0) vr += sc[SC_CB] * (double)f[(size_t)rb[tid] * T + tid];
    }
    S.vr[tid] = vr;
    f[(size_t)M.n * T + tid] = (VT)0;
    if constexpr (EXT)
      if (L.active[tid] && SW->nx[tid] > 0)
        ext_setup<T, NT>(M, L, *SW, *X, f, tid, ra[tid], rb[tid], w[tid], c ? c[tid] : 1.0);
  }
  __syncthreads();
  Vec<VT, LP> rr = vzero<VT, LP>(), ff = vzero<VT, LP>();
  // FP64 solves of a tile with a scenario in its first lane only: half the work
  // (in the wide CTAs, which take one scenario a tile)
  constexpr bool MAY_ONE = T == 2 && sizeof(VT) == 8 && NT > NTHREADS;
  const bool one = MAY_ONE && L.scen[T > 1 ? 1 : 0] < 0;
  if constexpr (MAY_ONE)
    if (one) red_forward<T, NT, 1, VT>(M, f, zt, part, rr, ff);
  if (!one) red_forward<T, NT, LP, VT>(M, f, zt, part, rr, ff);
#pragma unroll
  for (int off = 16; off >= TPR; off >>= 1)
#pragma unroll
    for (int j = 0; j < LP; ++j) {
      rr.v[j] += __shfl_xor_sync(0xffffffffu, rr.v[j], off);
      ff.v[j] += __shfl_xor_sync(0xffffffffu, ff.v[j], off);
    }
  if (wl < TPR)
#pragma unroll
    for (int j = 0; j < LP; ++j) {
      S.part[0][warp][g.lane + j] = (double)rr.v[j];
      S.part[1][warp][g.lane + j] = (double)ff.v[j];
    }
  __syncthreads();
  lap(1);
  // a warp per lane: the sparse dot products, the recurrence, and L^-1 v_m
  // added to the lane's vector
  const int t0 = M.tail_row0;
  for (int s = warp; s < T; s += NW) {
    double xa = 0.0;
    if (L.active[s] && !(hold && hold[s])) {
      RedScalars q{};
      double R = wl < NW ? S.part[0][wl][s] : 0.0, Z = wl < NW ? S.part[1][wl][s] : 0.0;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        R += __shfl_xor_sync(0xffffffffu, R, off);
        Z += __shfl_xor_sync(0xffffffffu, Z, off);
      }
      q.R = R;
      q.Z = Z;
      const int l = L.l[s];
      int e0 = 0, e1 = 0;
      if (l >= 0) {
        e0 = __ldg(M.br.ptr + l);
        e1 = __ldg(M.br.ptr + l + 1);
        const double* sc = M.br.sc + (size_t)l * SC_N;
        q.vy = __ldg(sc + SC_VY);
        q.my = __ldg(sc + SC_MY);
        q.vm2 = __ldg(sc + SC_VM2);
        q.w = __ldg(sc + SC_W);
        q.vr = S.vr[s];
        double u = 0.0, m0 = 0.0;
        for (int e = e0 + wl; e < e1; e += 32) {
          const int i = __ldg(M.br.row + e);
          const double x = (double)(i < t0 ? f[(size_t)i * T + s] : zt[(size_t)(i - t0) * T + s]);
          u = fma(__ldg(M.br.fv + e), x, u);
          m0 = fma(__ldg(M.br.fm + e), x, m0);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          u += __shfl_xor_sync(0xffffffffu, u, off);
          m0 += __shfl_xor_sync(0xffffffffu, m0, off);
        }
        q.u = u;
        q.m0 = m0;
      }
      auto place = [&](int i) {
        return i < t0 ? f + (size_t)i * T + s : zt + (size_t)(i - t0) * T + s;
      };
      bool done = false;
      if constexpr (EXT) {
        const int nx = SW->nx[s];
        if (nx > 0) {
          done = true;
          double x;
          const int its = ext_solve<T, NT>(M, L, *SW, *X, q, s, place,
                                           P.inner_rtol * P.inner_rtol, P.max_inner, x);
          xa = __shfl_sync(0xffffffffu, x, 0);
          const double xv = __shfl_sync(0xffffffffu, x, 1);
          if (wl >= 16 && wl < 16 + nx) X->xe[s][wl - 16] = x;
          if (xa != 0.0) {
            double kv = 0.0;  // the c_s' share of v
            for (int k = 0; k < nx; ++k) {
              const double xs = __shfl_sync(0xffffffffu, x, 2 + k) / xa;
              kv = fma(xs, X->k[s][k], kv);
              const int b = SW->xb[s][k], b1 = __ldg(M.bus.ptr + b + 1);
              for (int e = __ldg(M.bus.ptr + b) + wl; e < b1; e += 32) {
                VT* y = place(__ldg(M.bus.row + e));
                *y = (VT)fma(xs, __ldg(M.bus.f + e), (double)*y);
              }
              __syncwarp();
            }
            for (int e = e0 + wl; e < e1; e += 32) {
              VT* y = place(__ldg(M.br.row + e));
              *y = (VT)fma(xv / xa, __ldg(M.br.fm + e), fma(kv, __ldg(M.br.fv + e), (double)*y));
            }
          }
          if (wl == 0) iters[s] += its;
        }
      }
      if (!done) {
      double xb;
      const int its = reduced_cg(q, P.inner_rtol * P.inner_rtol, P.max_inner, xa, xb);
      if (xa != 0.0 && xb != 0.0) {
        const double k = xb / xa;
        for (int e = e0 + wl; e < e1; e += 32) {
          const int i = __ldg(M.br.row + e);
          VT* x = i < t0 ? f + (size_t)i * T + s : zt + (size_t)(i - t0) * T + s;
          *x = (VT)fma(k, __ldg(M.br.fm + e), (double)*x);
        }
      }
      if (wl == 0) iters[s] += its;
      }
    }
    if constexpr (EXT)
      if (xa == 0.0 && wl < KX) X->xe[s][wl] = 0.0;  // no step
    if (wl == 0) S.xa[s] = xa;
  }
  __syncthreads();
  lap(0);
  if constexpr (MAY_ONE)
    if (one) red_backward<T, NT, 1, VT>(M, f, zt, part);
  if (!one) red_backward<T, NT, LP, VT>(M, f, zt, part);
  if (M.ntblev == 0) __syncthreads();
  lap(2);
}

}  // namespace gpcg
