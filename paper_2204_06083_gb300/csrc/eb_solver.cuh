// Internal solver state: PCG scalars, work vectors and the AMG hierarchy.
#pragma once

#include <utility>
#include <vector>

#include "divide.cuh"
#include "eb_internal.cuh"

namespace ebk {

// Flexible CG (Polak-Ribiere beta): the x/r update also forms r.z_previous
// (the r'zold term) from the z still in place.  FIN_RRF: the batch's (r.r,
// r.z_previous) pairs, recorded per geometry; FIN_BETAF then takes r.z_previous
// from there; FIN_RZ0F is FIN_RZ0.  The single-grid PCG combines FIN_ALPHA and
// FIN_BETA inside its update kernels; the batch finalizes every op in its
// per-geometry kernel.
enum { FIN_INIT = 0, FIN_RZ0 = 1, FIN_ALPHA = 2, FIN_RR = 3, FIN_BETA = 4, FIN_RZ0F = 5, FIN_BETAF = 6, FIN_RRF = 7 };
enum { PCG_FLAG_NONFINITE = 1, PCG_FLAG_BREAKDOWN = 2 };
// what pcg_opts.profile times: the level-0 smoother launches, the learned stage's 32 -> 32
// convolutions, the level-1 (first coarse, CSR) smoother launches, the PCG's p update +
// apply launches (k_xpby_apply) or its x/r update launches (fused with the first level-0
// smoothing step when an AMG V-cycle follows)
enum { PROF_SMOOTHER = 1, PROF_CONV = 2, PROF_LEVEL1 = 3, PROF_XPBY = 4, PROF_UPDATE = 5 };

// rz[iters & 1] holds r'z of the current iteration; the kernel that computes
// the next one writes the other slot, so that no CTA reads a value another CTA
// of the same kernel is rewriting (the batch keeps using rz[0])
struct PcgScalars {
  double bb, rr, rz[2], pq, alpha, beta, tol2;
  int iters, flags, done;
  int maxit;  // iteration limit of the device-side loop (counted like iters)
  // iters & 1 as the x/r update of the iteration saw it: the r'z slot of the
  // p update, whose launch may also advance iters (device-side loop)
  int slot;
  double rzo;  // batched flexible PCG: r'zold of the iteration (FIN_RRF)
  double* x;   // the vector the solve updates: captured iterations serve any
};

struct Hierarchy;  // AMG levels (amg.cu)
struct OpParams;   // operator constants of the PCG kernels (eb_solve.cu)

struct Solver {
  EBHandle* eb = nullptr;
  // stream the solver's memory belongs to (set at setup); destroying a solver
  // never reads *eb, which may already be gone
  cudaStream_t home = 0;
  double shift = 0.0;
  amg_opts opts{};
  Hierarchy* H = nullptr;
  double setup_ms = 0.0;
  int csr_epl = 2;  // CSR kernels of the V-cycle: target entries per lane of a row group (amg_tune_csr)
  // full-grid work vectors (touched on the active tiles only)
  double *r = nullptr, *z = nullptr, *p = nullptr, *q = nullptr, *tmp = nullptr;
  double* wx = nullptr;  // the implicit wave step's solution vector (allocated on first use)
  bool flexible() const { return H != nullptr && (opts.vcycle_prec == EB_F32 || opts.vcycle_prec == EB_BF16); }
  // the flexible (Polak-Ribiere) beta: reduced-precision V-cycle or learned stage
  bool flex_for(int kind) const { return kind == EB_PC_AMG_NN || (kind == EB_PC_AMG && flexible()); }
  nn_handle* nn = nullptr;  // learned stage of EB_PC_AMG_NN (set for one solve)
  int nn_mode = 0;          // eb_nn_mode of that stage
  // reduction partials: [p'q | r'r] regions of 2 npart each, then the r'z region
  // (nblk partials from the PCG's own dot kernel, one per CTA of the V-cycle's
  // last smoothing launch), then the r'zold region of npart
  int npart = 1;  // max(nblk, nblk_iter() of the FP64 iteration, which has no fewer CTAs than the DF one)
  double* part = nullptr;
  double* part_pq() const { return part; }
  double* part_rr() const { return part + 2 * (int64_t)npart; }
  double* part_rz() const { return part + 4 * (int64_t)npart; }
  // r'zold partials of the flexible beta (from the x/r update)
  double* part_rzo() const { return part + 4 * (int64_t)npart + rz_cap; }
  // CTAs (= partials) of the iteration's x/r update and p update + apply
  // (a full grid leaves room for the CTA of the loop test, so that all are
  // resident at once)
  int nblk_iter() const { return std::min(list_blocks(eb->num_pairs, iter_threads()), 4 * num_sms() - 1); }
  int iter_threads() const { return df_on ? list_threads_df(eb->num_pairs) : list_threads(eb->num_pairs); }
  int64_t rz_cap = 0;
  int nblk = 1;
  int rz_n = 1;  // r'z partials written by the last precondition()
  PcgScalars* sc = nullptr;
  // not page-locked: that allocation and its release (which waits for the
  // device) cost 320 us per solver, its copies of ~0.2 KB no more than these
  PcgScalars sc_host{};
  int64_t nlaunch = 0;  // kernel launches issued (reported per solve)
  // event timing of the level-0 smoother launches
  bool prof_on = false;
  int prof_what = PROF_SMOOTHER;
  int prof_n = 0;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_ev;
  double prof_acc_ms = 0.0;
  int prof_acc_n = 0;
  // captured PCG iteration (CUDA graph), keyed by what it depends on: neither b
  // nor x, whose address the iteration takes from sc, but the state of the
  // learned stage (nn_stage_state), whose buffers and route it holds
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t gexec = nullptr;
  uint64_t g_nn = 0;
  int g_tile_gen = -1;
  int g_nn_mode = -1;
  int g_iters = 0, g_kind = -1, g_prof = -1, g_pairs = 0;
  int64_t g_launches = 0;
  // the whole iteration loop on the device: a conditional WHILE node whose
  // body is one iteration (no host round trip per iteration)
  cudaGraphExec_t lexec = nullptr;
  int l_kind = -1, l_nn_mode = -1, l_tile_gen = -1;
  uint64_t l_nn = 0;
  int64_t l_launches = 0;  // kernel launches per loop iteration
  // the DF outer iteration (pcg_opts.outer_prec = EB_DF64) for the current
  // solve: x, r, p, q hold double-float pairs (x in xdf), z FP32; diag_df is
  // the DF copy of the cut CPs' D_k (built on first use)
  bool df_on = false;
  float2* diag_df = nullptr;
  float2* beta_df[3] = {nullptr, nullptr, nullptr};  // DF copies of beta per axis (variable coefficient)
  int df_gen = -1;  // the handle's tile_gen the DF copies were built for
  // outer precision of the solves without their own options: heat_step,
  // wave_theta_step, pcg_solve with NULL opts (amg_set_outer_prec)
  int outer_default = EB_F64;
  int default_outer() const;
  // level-0 smoothing steps of batched 2D views through tensor copies (on by
  // default; batch_set_level0_tma), and the device flag their bounded waits set
  bool l0_tma = true;
  int* dev_err = nullptr;
  double* xdf = nullptr;  // the DF image of x (tmp may hold the right-hand side)
  int g_df = -1, l_df = -1;

  void alloc_work(cudaStream_t s);
  void free_work();
  void finalize(int op, const double* src, cudaStream_t s, int count = -1);  // count < 0: nblk partials
  // first_done: amg_update_first did the V-cycle's first level-0 step for r
  void precondition(int kind, const double* r, double* z, cudaStream_t s, bool first_done = false);
  int pcg(const double* b, double* x, double rtol, int maxit, const pcg_opts& o, pcg_stats* stats, cudaStream_t s);
  int heat(double dt, double theta, const double* b1, const double* b0, double* u, double rtol, int maxit,
           pcg_stats* stats, cudaStream_t s);
  int wave_theta(double dt, double theta, double* ua, double* ub, int nsteps, double rtol, int maxit,
                 pcg_stats* stats, cudaStream_t s);
  void prof_begin(int mode, cudaStream_t s);
  void prof_mark(cudaStream_t s, bool start, int what = PROF_SMOOTHER);
  void prof_collect(int first, int count);
  void prof_end(pcg_stats* st, cudaStream_t s);
  void prof_release();
  // cond: inside the device-side loop, the handle its last launch sets
  void iteration(int kind, cudaStream_t s, const cudaGraphConditionalHandle* cond = nullptr);
  // p = z + beta p and q = h^2 (sigma I + A) z + beta q with the p.q partials
  // (eb_solve.cu); flex: the Polak-Ribiere beta (r'zold partials in part_rzo)
  void xpby_apply(const OpParams& op, bool flex, int first, cudaStream_t s,
                  const cudaGraphConditionalHandle* cond = nullptr);
  void graph_prepare(int kind, int iters, int profile, cudaStream_t s);
  void graph_release();
  void loop_prepare(int kind);
  void loop_release();
};

// Instantiates { while (condition) body } as one executable graph: body(st,
// h) enqueues one pass on the capture stream st and must end with a kernel
// that sets the condition handle h (cudaGraphSetConditional); the condition
// starts at 1.  cap is a non-blocking stream used only for the capture.
cudaGraphExec_t build_while_graph(cudaStream_t cap,
                                  const std::function<void(cudaStream_t, cudaGraphConditionalHandle)>& body);

// AMG (amg.cu)
void amg_build(Solver& S, cudaStream_t s);
void amg_free(Solver& S);
// Sum of v over the CTA: through shared memory, one warp adding the columns
// and then its lanes; thread 0 holds the result.  Every reduction partial of
// the PCG is formed this way.  GB300 issues 0.4 FP64 lanes per clock and
// scheduler, so a warp-wide FP64 addition occupies one for 80 clocks: a CTA of
// 256 threads spends 12 of them here, where shuffle trees in all its warps and
// a serial end take 48.  sm: blockDim.x doubles.
__device__ __forceinline__ double warp_column_sum(const double* sm, int n) {
  double s = sm[threadIdx.x & 31];
  for (int i = (threadIdx.x & 31) + 32; i < n; i += 32) s += sm[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

__device__ __forceinline__ double block_sum(double v, double* sm) {
  __syncthreads();
  sm[threadIdx.x] = v;
  __syncthreads();
  return threadIdx.x < 32 ? warp_column_sum(sm, (int)blockDim.x) : 0.0;
}

// What a CTA of the update kernels needs of the scalars, read by its thread 0 at
// the start, all loads at once, ahead of the partial sums.  done is passed on
// through shared memory: another CTA of the launch may set it meanwhile, and
// threads that read it themselves could disagree, part of the CTA skipping the
// barriers the rest waits at.
struct PcgHead {
  int done = 0, k = 0;  // k: the iteration's r'z slot
  double rz = 0.0;
};
__device__ __forceinline__ PcgHead pcg_head(const PcgScalars* sc, bool recorded_slot) {
  PcgHead h;
  if (threadIdx.x == 0) {
    const volatile PcgScalars* v = sc;
    const int it = v->iters, sl = v->slot;
    const double a = v->rz[0], b = v->rz[1];
    h.done = v->done;
    h.k = recorded_slot ? sl : (it & 1);
    h.rz = h.k ? b : a;
  }
  return h;
}

// sum of n partials in a fixed order, the same in every CTA of a launch;
// thread 0 holds the result.  Four warps load (as many as the FP64 additions
// keep busy: every CTA repeats the sum), one combines.  sm: 128 doubles.
__device__ __forceinline__ double sum_parts(const double* part, int n, double* sm) {
  const int w = min((int)blockDim.x, 128);
  double a = 0.0;
  if ((int)threadIdx.x < w) {
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += w) a += part[i];
  }
  __syncthreads();
  if ((int)threadIdx.x < w) sm[threadIdx.x] = a;
  __syncthreads();
  return threadIdx.x < 32 ? warp_column_sum(sm, w) : 0.0;
}

// two such sums side by side, by the two halves of the CTA (blockDim.x >= 64);
// thread 0 holds both.  sm: 258 doubles.
__device__ __forceinline__ void sum_parts2(const double* pa, int na, const double* pb, int nb, double* sm, double& a,
                                           double& b) {
  const int half = (int)blockDim.x >> 1, g = (int)threadIdx.x >= half, l = (int)threadIdx.x - g * half;
  const int w = min(half, 128), n = g ? nb : na;
  const double* p = g ? pb : pa;
  double v = 0.0;
  if (l < w) {
#pragma unroll 4
    for (int i = l; i < n; i += w) v += p[i];
  }
  __syncthreads();
  if (l < w) sm[128 * g + l] = v;
  __syncthreads();
  if (l < 32) {
    const double s = warp_column_sum(sm + 128 * g, w);
    if (l == 0) sm[256 + g] = s;
  }
  __syncthreads();
  a = sm[256];
  b = sm[257];
}

// into L1 ahead of a load (the reduction sums between hide the latency)
__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// alpha = rz / p'q from the nblk partials of k_xpby_apply (q scaled by h^2: the
// CG step length over h^2), formed by every CTA in the same order; CTA 0 records
// p'q, alpha and a breakdown (p'q <= 0 or not finite).  Thread 0's part, given
// the summed p'q
__device__ __forceinline__ double pcg_alpha_from(PcgScalars* sc, const PcgHead& h, double pq) {
  const bool ok = pq > 0.0;  // false for NaN too
  const double alpha = ok ? h.rz / pq : 0.0;
  if (blockIdx.x == 0) {
    sc->pq = pq;
    sc->alpha = alpha;
    sc->slot = h.k;
    if (!ok) {
      sc->flags |= isfinite(pq) ? PCG_FLAG_BREAKDOWN : PCG_FLAG_NONFINITE;
      sc->done = 1;
    }
  }
  return alpha;
}

// all threads of the CTA; false (all threads) when the solve is done
__device__ __forceinline__ bool pcg_alpha(PcgScalars* sc, const double* pq_part, int nblk, double* sm, double& alpha) {
  __shared__ double s_alpha;
  __shared__ int s_done;
  const PcgHead h = pcg_head(sc, false);
  const double pq = sum_parts(pq_part, nblk, sm);
  if (threadIdx.x == 0) {
    s_done = h.done;
    if (!h.done) s_alpha = pcg_alpha_from(sc, h, pq);
  }
  __syncthreads();
  alpha = s_alpha;
  return s_done == 0;
}

// 2^-600 <= |x| < 2^600, by the exponent bits
__device__ __forceinline__ bool pcg_mid_range(double x) {
  return (uint32_t)((__double2hiint(x) >> 20 & 0x7ff) - (1023 - 600)) < 1200u;
}

// The end of an iteration, thread 0's part: beta = (v - t) / rz from the summed
// r'z (v) and, flexible, r'zold (t); with rec (one CTA of the launch) recorded
// with the next r'z and a breakdown.  inv_rz: 1 / h.rz, formed ahead; the
// quotient is that of a division (div_by), and one where the reciprocal or the
// correction would leave FP64's normal range (r'z of a tiny right-hand side).
__device__ __forceinline__ double pcg_beta_from(PcgScalars* sc, const PcgHead& h, double inv_rz, double v, double t,
                                                bool rec) {
  const bool ok = v > 0.0;
  const double num = v - t;
  const bool mid = pcg_mid_range(h.rz) && pcg_mid_range(num);
  const double beta = !ok ? 0.0 : mid ? div_by(num, DivBy<double>{h.rz, inv_rz}) : num / h.rz;
  if (rec) {
    sc->beta = beta;
    sc->rz[h.k ^ 1] = v;
    if (!ok) {
      sc->flags |= isfinite(v) ? PCG_FLAG_BREAKDOWN : PCG_FLAG_NONFINITE;
      sc->done = 1;
    }
  }
  return beta;
}

// The device-side loop's test (one thread), after the beta breakdown check: r'r
// of this iteration's update (v), then continue while not converged (or broken
// down) and below the iteration limit.  CTAs that start after it and see done
// skip the p, q update, which a finished loop does not use.
__device__ __forceinline__ void pcg_loop_test(PcgScalars* sc, double v, cudaGraphConditionalHandle h) {
  if (!sc->done) {
    sc->rr = v;
    sc->iters += 1;
    if (!isfinite(v)) {
      sc->flags |= PCG_FLAG_NONFINITE;
      sc->done = 1;
    } else if (v <= sc->tol2 * sc->bb) {
      sc->done = 1;
    }
  }
  cudaGraphSetConditional(h, (!sc->done && sc->iters < sc->maxit) ? 1u : 0u);
}

// The PCG update x += alpha p, r -= alpha q (with the r'r partials of
// k_update_xr) fused with the first level-0 smoothing step of the V-cycle that
// follows (which then starts at its second step); 0 if the hierarchy has no
// such step (a single level), else the launch was issued.
struct PcgUpdate {
  PcgScalars* sc = nullptr;
  double* r = nullptr;  // x is sc->x
  const double *p = nullptr, *q = nullptr, *pq_part = nullptr;
  int nblk = 0;
  double* rr_part = nullptr;
  double h2 = 1.0;  // q holds h2 (sigma I + A) p: x takes the step alpha h2
  // flexible CG: partials of (new r).z with the z still in z (r'zold)
  const double* z = nullptr;
  double* rzo_part = nullptr;
  // the DF outer iteration: x, r, p, q hold double-float pairs, z FP32
  bool df = false;
};
int amg_update_first(Solver& S, const PcgUpdate& u, cudaStream_t s);

// The batched DF iteration's x/r update with the V-cycle's first level-0 step
// (a hierarchy of two or more levels with FP32 or BF16 storage); x is sc[0].x
struct BatchUpdate {
  const int32_t* tile_geo = nullptr;
  const PcgScalars* sc = nullptr;
  double* r = nullptr;
  const double *p = nullptr, *q = nullptr;
  const float* z = nullptr;
  double* part = nullptr;  // per-tile pairs (r.r, r.zold)
};
void amg_batch_update_first(Solver& S, const BatchUpdate& u, unsigned grid, cudaStream_t s);

// z = V r.  With dot, the last level-0 smoothing launch also writes per-CTA
// partials of r.z to dot->part; returns their count, or 0 if no launch wrote
// them (single-level hierarchy), in which case the caller computes the dot
// itself.
struct VcycleDot {
  const double* r = nullptr;
  double* part = nullptr;
  // the DF outer iteration: r holds double-float pairs, z is written in FP32
  // (part null: no partials, z on every node of the active tiles)
  bool df = false;
  double* tile_part = nullptr;  // batched DF iteration: per-tile pairs (r.z, 0)
};
// first_done: amg_update_first already did the first level-0 step for this r.
int amg_vcycle_grid(Solver& S, const double* r, double* z, cudaStream_t s, const VcycleDot* dot = nullptr,
                    bool first_done = false);
void amg_fill_info(const Solver& S, amg_info_t* out);
int amg_levels(const Solver& S);  // levels of the hierarchy (0 without one)
void amg_copy_level(const Solver& S, int level, int which, int32_t* rowptr, int32_t* col, double* val, cudaStream_t s);

// learned stage (cnn.cu): a number that no other handle has or had and that
// changes with everything a captured stage depends on (0: no stage)
uint64_t nn_stage_state(const nn_handle* nn);
// buffers for grids of eb's size (before any capture),
// then z <- z + omega h^2 rms(s) N(s / rms(s), m), s = r - (shift I + A) z
void nn_stage_prepare(nn_handle* nn, const EBHandle& eb, cudaStream_t s);
void nn_stage_apply(nn_handle* nn, const EBHandle& eb, double shift, int mode, const double* r, double* z,
                    int64_t& nlaunch, Solver* prof, cudaStream_t s);

}  // namespace ebk

// the opaque AMG / solver handle of the C ABI
struct amg_handle {
  ebk::Solver s;
};
