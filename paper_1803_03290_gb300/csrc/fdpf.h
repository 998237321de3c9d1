// Parameters and launchers of the persistent N-1 kernel (fdpf.cu).
#pragma once
#include <algorithm>

#include "common.cuh"

namespace gpcg {

#ifndef FDPF_NTHREADS
#define FDPF_NTHREADS 256
#endif
constexpr int NTHREADS = FDPF_NTHREADS;  // threads per CTA of the persistent kernel
constexpr double DIVERGE_LIMIT = 1.0e4;   // p.u.: a larger mismatch is divergence
constexpr double DIVERGE_GROWTH = 10.0;   // as is growth to this multiple of the best
enum { PREC_IC0 = 0, PREC_JACOBI = 1, PREC_EXACT = 2 };

constexpr int MD_DEG = 0xff, MD_TYPE_SHIFT = 8, MD_TYPE = 3, MD_OVER = 1 << 10;

// The buses of a half-step in the order its mismatch and update passes visit
// them, with what they need to know of each in that order, so that a warp's
// loads coalesce: md = {bus, preorder, degree in the padded adjacency (MD_DEG)
// | bus type | MD_OVER: overflow entries, row of the half-step's matrix}, the
// neighbour and (c g, c b_y) of each slot (slot a of entry k at a * n + k), the
// admittance diagonal and the scheduled injections.  Bus order, sorted by
// degree and type inside windows of MD_WINDOW entries: the threads of a warp
// run neighbour loops of equal length.
constexpr int MD_WINDOW = 512;
struct BusTab {
  const int4* md = nullptr;
  const int32_t* nbr = nullptr;
  const double2 *gb = nullptr, *yd = nullptr, *pq = nullptr;
  int n = 0;
};

struct FdpfParams {
  DevGrid G;
  int S = 0, n_tiles = 0;
  int fill = 0;                // lanes of a tile that take scenarios (at most T)
  ScenInfo sc;
  const double *th0 = nullptr, *V0 = nullptr;  // warm start (bus order)
  const double *c0 = nullptr, *s0 = nullptr;   // cos, sin of th0
  const double2* ef0 = nullptr;                // V0 (c0, s0)
  const double *r0P = nullptr, *r0Q = nullptr; // base-case mismatch per bus (null: not used)
  int flat_start = 0;
  double tol = 1e-4, inner_rtol = 3e-3;
  int max_outer = 50, max_inner = 500, precond = PREC_EXACT;
  int reduced = 0;  // the inner solves in their reduced form (reduced_form below)
  int32_t* tile_counter = nullptr;     // scenario queue head
  const int32_t* order = nullptr;      // scenarios in processing order (null: 0..S-1)
  void *wx = nullptr, *wr = nullptr, *wp = nullptr, *wq = nullptr, *wz = nullptr;
  size_t vstride = 0;  // elements per slot of one vector
  // FP64 state per slot: theta, and e + jf interleaved over the we and wf
  // regions together ([slot][bus][lane][e, f], 2 sstride per slot); the
  // persistent N-1 kernel keeps no |V| (|e + jf|), so wV is scratch for the
  // DC and adjoint kernels only
  double *wth = nullptr, *wV = nullptr, *we = nullptr, *wf = nullptr;
  size_t sstride = 0;  // elements per slot of one state array
  double *out_theta = nullptr, *out_vm = nullptr, *out_flow = nullptr, *out_maxload = nullptr;
  // output column -> internal bus (null: identity): the outputs are written
  // column by column, so neighbouring threads store neighbouring columns
  const int32_t* out_bus_map = nullptr;
  int32_t *out_iters = nullptr, *out_status = nullptr;
  // overload screen: per scenario the number of branches loaded above their
  // rating, and those branches as a bit mask of mask_words words
  int32_t* out_nover = nullptr;
  uint32_t* out_ovmask = nullptr;
  // diagnostics, or null: [8] per-phase SM cycles summed over CTAs, then per
  // scenario the global timer (ns) when a lane took it and when it retired
  unsigned long long* phase_cycles = nullptr;
  BusTab tabP, tabQ;  // non-slack buses, rows of B'; PQ buses, rows of B''
};

// Whether a screen's inner solves run in their reduced form (reduced.cuh): the
// complete base-case factor in the precision of the vectors, and for FP32 vectors
// an outer tolerance that leaves nothing of their rounding in the results.
//
// At a loose tolerance a state ends one inner solve away from the last
// mismatch that failed it, and with FP32 vectors that solve is rounded in the
// fourth digit: the PCG's recursive residual asks for one more iteration in 5 %
// of the scenarios than the reduced recurrence does.  Both states meet the
// tolerance, but a branch within 1e-4 of its rating may be overloaded in one and
// not in the other, and a scenario without a solution ends wherever the rounding
// takes it.  A verdict would then depend on which kernel the preconditioner and
// the list allow.  Overload masks against the PCG's, at 1e-4 p.u.: different in 1
// of 20 lists of 13,500 outages of 10,000 buses and 1 of 25 of 2,700 outages of
// 2,000 buses with reactive limits (converged scenarios), and in 1 of 10 of 2,047
// outages of 50,000 buses (scenarios that do not converge).  So FP32 screens keep
// the PCG there, at its price: 13,500 outages of 10,000 buses 73.3 ms (reduced
// 42.4), 2,047 of 50,000 buses 98.5 ms (57), 2,700 of 2,000 buses with limits
// 38.6 ms (13.5).  From 1e-9 p.u. down the results agree to 1e-9 and the verdicts
// with them; FP64 vectors take the same iterations in either form.
constexpr double REDUCED_F32_TOL = 1e-9;
template <typename VT>
inline bool reduced_form(int precond, const DevMatT<VT>& MP, const DevMatT<VT>& MQ,
                         double tol = 0.0) {
  return precond == PREC_EXACT && MP.br.ptr && MQ.br.ptr && !MP.Lh && !MQ.Lh &&
         (sizeof(VT) == 8 || tol <= REDUCED_F32_TOL);
}

// A launch of S scenarios too few to fill the GPU: threads per CTA, CTAs and
// lanes per tile (tiles of two, reduced inner solves without extension rows).
// A pass over the rows then lasts as long as its chain of loads times the rows
// per thread, so the threads that other tiles do not need go to this one; and
// while there are SMs to spare a tile takes one scenario, which halves the FP64
// work an SM has to do for it.
struct WideLaunch {
  int nt, grid, fill;
};
// Dynamic shared memory a wide CTA takes for the vector of its solves (the
// substitutions' gathers then wait on shared memory), 0 if the vector does not
// fit: what one CTA of 1,024 threads or two of 512 leave of the SM's shared memory
// beside the kernel's own arrays (27.8 KB for FP64 and 1,024 threads), as the
// device and the kernel report it.
template <typename VT>
size_t wide_shared(int nt, size_t vec_bytes);
// Grids of fewer rows than threads gain nothing (FP64 solves do from 512: the
// dense tail's terms are split over the threads).  Kernel times for tolerance
// 1e-10, CTAs of 256 / 512 / 1,024 threads: 97 outages of a 2,000-bus grid 2.04 /
// 1.58 / 1.48 ms (one scenario a tile; two: - / 1.76 / 1.65), 300 outages 2.02 / 1.75
// / 1.65 ms, 600 outages 3.72 / 2.89 / 3.06 ms, 1,000 outages 4.04 / 3.46 / 4.98 ms,
// 2,700 outages 6.9 / 8.1 / 12.1 ms; 10,000 buses, 1,000 outages 16.1 / 13.7 / 16.3 ms,
// 1,500 outages 18.2 / 20.1 / 23.2 ms; 180 outages of 120 buses 1.57 / 1.82 /
// 2.07 ms.
inline WideLaunch wide_launch(int S, int num_sms, int rows, bool fp64) {
  const int most = rows >= 1024 ? 1024 : rows >= 512 || fp64 ? 512 : NTHREADS;
  const WideLaunch w = S <= num_sms       ? WideLaunch{std::min(1024, most), S, 1}
                       : S <= 2 * num_sms ? WideLaunch{std::min(1024, most), (S + 1) / 2, 2}
                       : S <= 8 * num_sms
                           ? WideLaunch{std::min(512, most), std::min((S + 1) / 2, 2 * num_sms), 2}
                                          : WideLaunch{NTHREADS, 0, 2};
  return w.nt == NTHREADS ? WideLaunch{NTHREADS, 0, 2} : w;
}

// The persistent N-1 kernel for tiles of T scenarios (2 to 32; generator
// outages, P.sc.gen_bus set: 2, 4 or 8) on `grid` slots.  zbytes > 0 (branch
// outages without reactive limits, T = 2 or 4): each tile's z vector in
// zbytes of dynamic shared memory, P.wz unused.
template <typename VT>
cudaError_t launch_fdpf(cudaStream_t st, int T, int grid, const FdpfParams& P,
                        const DevMatT<VT>& MP, const DevMatT<VT>& MQ, size_t zbytes = 0,
                        int nt = NTHREADS, size_t wide_bytes = 0);
template <typename VT>
int fdpf_max_blocks_per_sm(int T, bool gen, size_t zbytes, bool red);
// the generator-outage kernel (fdpf_gen.cu)
template <typename VT>
cudaError_t launch_fdpf_gen(cudaStream_t st, int T, int grid, const FdpfParams& P,
                            const DevMatT<VT>& MP, const DevMatT<VT>& MQ);
template <typename VT>
int fdpf_blocks_gen(int T, bool red);
template <typename VT>
cudaError_t launch_apply(cudaStream_t st, int grid, const DevMatT<VT>& M, int op, int S,
                         const int32_t* outages, const int32_t* f, const int32_t* t,
                         const double* X, double* Y, VT* wbuf, size_t vstride, int precond);
cudaError_t launch_base_trig(cudaStream_t st, int n, const double* th, const double* V, double* c,
                             double* s, double2* ef);
cudaError_t launch_base_residual(cudaStream_t st, const DevGrid& G, const double* V0,
                                 const double* c0, const double* s0, double* r0P, double* r0Q);

// plain.cu: the unbatched FP64 path, one scenario per cooperative launch
// over the whole GPU.  Work buffers, device memory owned by the caller.
struct PlainBuffers {
  double* part = nullptr;          // [2 * 4 * grid]
  unsigned int* bar = nullptr;     // [2], zero before the first launch
  int* err = nullptr;              // [1], zero before the first launch
  unsigned wait_limit = 1u << 25;  // polls of a barrier wait (~64 ns each) before it gives up
  double *x = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *z = nullptr, *t = nullptr;
  double *th = nullptr, *V = nullptr, *ef = nullptr;  // [n], [n], [2 n]
};
cudaError_t launch_plain(cudaStream_t st, int grid, const FdpfParams& P,
                         const DevMatT<double>& MP, const DevMatT<double>& MQ,
                         const PlainBuffers& B, int s);
int plain_grid(int num_sms);  // CTAs of the cooperative launch (0: not available)

// adjoint.cu
struct AdjParamsView {
  const double* P;   // [n] injections, internal bus order
  const double* b;   // [m] branch susceptances
  double *gP, *gb, *loss;  // per-slot sums: [slots][n], [slots][m], [slots]
  double* g;               // [slots][m][2] scratch: dL/df of a slot's scenarios
};
cudaError_t launch_adjoint(cudaStream_t st, int grid, const FdpfParams& P, const AdjParamsView& A,
                           const DevMatT<double>& M);
int adjoint_max_blocks_per_sm(bool red);

// Inputs and outputs of the DC (P-theta) quick screen.
struct DcParamsView {
  const double* P;              // [n] injections, internal bus order
  const int32_t* user_of_bus;   // internal bus -> caller's index
  double* theta;                // [S][n] caller's bus order, or null
  double* flow;                 // [S][m], or null
  double* maxload;              // [S], or null
  int32_t* iters;               // [S] PCG iterations, or null
  int32_t* status;              // [S], or null
  int32_t* nover;               // [S] branches loaded above their rating, or null
  uint32_t* ovmask;             // [S][(m + 31) / 32] those branches as bits, or null
  const int2* row_pre;          // [n] caller's bus -> row of B' (-1: slack), preorder
  const int2* br_rows;          // [m] rows of B' of the from and the to end
};
template <typename VT>
cudaError_t launch_dc(cudaStream_t st, int grid, const FdpfParams& P, const DcParamsView& D,
                      const DevMatT<VT>& M, const DevMatT<double>& M64);
template <typename VT>
int dc_max_blocks_per_sm();
// The same for the complete factor with FP64 solves and no iteration counts
// asked for; f0: 2 (rows + 1) doubles of scratch.
cudaError_t launch_dc_direct(cudaStream_t st, int grid, const FdpfParams& P,
                             const DcParamsView& D, const DevMatT<double>& M, double* f0);
int dc_direct_max_blocks_per_sm();
cudaError_t launch_slot_sum(cudaStream_t st, int n, int slots, const double* acc,
                            const int32_t* map, double* out);
cudaError_t launch_gather_perm(cudaStream_t st, int n, const int32_t* idx, const double* src,
                               double* dst);

}  // namespace gpcg
