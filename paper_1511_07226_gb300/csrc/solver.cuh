// Method interface shared by the solver drivers (internal).
#pragma once

#include "pfk_internal.cuh"

namespace pfk {

// Everything a method's kernels need besides its own vectors.
struct SolveEnv {
  pfk_context* ctx;
  const pfk_operator* op;
  const pfk_pc* pc;          // null = identity
  cudaStream_t st;
  SolveCtl* ctl;             // device control block
  double* partials;          // reduction partials of the method's kernels
  int64_t partials_cap;      // doubles available at `partials`
  int64_t N;

  // True if a launch of `blocks` blocks writing `stride` partials each fits.
  bool partials_fit(int blocks, int stride) const { return (int64_t)blocks * stride <= partials_cap; }
  // The same for a two-level combine (block rows plus one row per group).
  bool partials_fit_2l(int blocks, int stride) const {
    return blocks <= kCombineGroup * kMaxCombineGroups &&
           (int64_t)(blocks + (blocks + kCombineGroup - 1) / kCombineGroup) * stride <= partials_cap;
  }
  cudaEvent_t pass_ev0, pass_ev1;   // profiling: recorded around the fused pass (or null)
  // How the preconditioner adds and waits.  pinned (a pipelined method, or a
  // preconditioner in reduced precision) holds for the method's own sums too.
  PcCall pcc;

  // out = add + B(v); B = identity when pc is null.
  cudaError_t pc_apply(const double* v, double* out, const double* add, const int* status) const;
  // Records pass_ev0 (which = 0) or pass_ev1 (1) if profiling.
  cudaError_t mark_pass(int which) const;
};

// A Krylov method as a pipeline fill plus a replayable iteration.
class Method {
 public:
  virtual ~Method() {}
  // FP64 words of workspace for n unknowns and window/restart length mmax.
  virtual int64_t workspace_doubles(int64_t N, int mmax) const = 0;
  virtual void bind(double* ws, int64_t N, int mmax) = 0;
  // One length-N vector the driver may use between phases (true residual).
  virtual double* scratch() = 0;
  // (Re)start from x: pipeline fill and the scalars of iteration 0; sets ctl->status.
  virtual cudaError_t fill(const SolveEnv& env, const double* b, double* x) = 0;
  // One iteration; every kernel is a no-op once ctl->status != kRun.
  virtual cudaError_t iteration(const SolveEnv& env, double* x) = 0;
  // Called by the driver when an iteration group stopped with status kRun at
  // the end of a restart cycle (GMRES types); default: nothing.
  virtual cudaError_t end_cycle(const SolveEnv& env, double* x) { (void)env; (void)x; return cudaSuccess; }
  // Iterations one call of iteration() covers at most.
  virtual int iterations_per_step() const { return 1; }
  // Whether u_i, p_i and s_i are formed from r_i and u_i themselves (FCG, GCR,
  // FGMRES): with a preconditioner in FP64 a rounding difference of the inner
  // products then stays one (up to 5e-15 over 130 drawn problems).  In the
  // pipelined recurrences, where no vector is ever formed anew, it grows: by up
  // to 1e8 in 20 iterations of PIPEGCR at 26^3, contrast 1e3.  And a
  // preconditioner that rounds its input to FP32 turns it into a difference of
  // 6e-8 in the entries that round the other way (FGMRES with the BF16
  // smoother, 118 x 112 x 127, 25 iterations: 8.5e-10 in the solution).
  virtual bool blocking() const { return false; }
  // Number of ring/Hessenberg columns (GMRES types restart after this many).
  virtual int cycle_length() const { return 0; }
  // Once per solve, before bind: picks the persistent single-launch form when
  // the method has one, the problem is eligible and `mode` allows it (0 auto,
  // 1 never, 2 required).  Returns whether it did.
  virtual bool configure(const pfk_context* ctx, const pfk_operator* op, const pfk_pc* pc, int64_t N, int mode) {
    (void)ctx; (void)op; (void)pc; (void)N; (void)mode;
    return false;
  }
  // Once per solve, before the graphs are captured (e.g. the PIPEFGMRES shift
  // estimate); may synchronise.  `dscalar` is a device scalar slot; the method
  // reports the shift it uses (NaN if none) in *host_sigma.
  virtual cudaError_t prepare(const SolveEnv& env, const double* b, double* dscalar, double* host_sigma) {
    (void)env; (void)b; (void)dscalar;
    *host_sigma = NAN;
    return cudaSuccess;
  }
};

// Window dots, the reduction of the CR types and the base methods: one
// register accumulator per window slot and thread (independent FMAs, the
// loads of a whole window in flight), then warp_sum_transposed: lane l returns
// the warp's <v, s_j> for j = l / (32 / NW).  s_off holds the slots' offsets.
// body(e, v_e) adds the caller's own products.  The loop is instantiated for
// window sizes rounded up to 4: with one loop for 32 slots the guarded products
// of the empty slots were issued all the same (101x97x93: 79 us at every window
// size; PIPEGCR at 64^3: 45 us at the median window and 63 at the largest, now 35
// and 43).  The order of a thread's sum depends on the grid alone.
constexpr int kWinThreads = 128;
constexpr int kWinBlocksPerSm = 4;   // base methods: 128 registers

template <int NR, bool LEAN, int NW, typename F>
__device__ __forceinline__ void window_dots_loop(const double* __restrict__ v, const double* __restrict__ S,
                                                 const size_t* s_off, int nu, int64_t N, double (&acc)[NW],
                                                 F&& body) {
  for (int64_t e = (int64_t)blockIdx.x * kWinThreads + threadIdx.x; e < N; e += (int64_t)gridDim.x * kWinThreads) {
    const double ve = __ldg(&v[e]);
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      // rows below NR - 3 exist; the last ones may not
      if constexpr (LEAN) {
        if (j < nu) acc[j] = fma(ve, __ldg(&S[s_off[j] + e]), acc[j]);
      } else {
        const double sv = (j < NR - 3 || j < nu) ? __ldg(&S[s_off[j] + e]) : 0.0;
        acc[j] = fma(ve, sv, acc[j]);
      }
    }
    body(e, ve);
  }
}

// LEAN: every slot guarded, which keeps fewer loads in flight and so fewer
// registers; for the sizes above 16, in a kernel held to 96 registers (without
// it 750 bytes of spills).
template <int NR, bool LEAN, int NW, typename F>
__device__ __forceinline__ double window_dots_n(const double* __restrict__ v, const double* __restrict__ S,
                                                const size_t* s_off, int nu, int64_t N, F&& body) {
  double acc[NW];
#pragma unroll
  for (int j = 0; j < NW; ++j) acc[j] = 0.0;
  if constexpr (LEAN) asm("" : "+r"(nu));   // or the branch's lower bound on nu removes the guards
  window_dots_loop<NR, LEAN>(v, S, s_off, nu, N, acc, body);
  return warp_sum_transposed<NW>(acc);
}

template <int NW, bool LEAN = false, typename F>
__device__ __forceinline__ double window_dots(const double* __restrict__ v, const double* __restrict__ S,
                                            const size_t* s_off, int nu, int64_t N, F&& body) {
  if (nu <= 4) return window_dots_n<4, false, NW>(v, S, s_off, nu, N, body);
  if (nu <= 8 || NW == 8) return window_dots_n<8, false, NW>(v, S, s_off, nu, N, body);
  if constexpr (NW >= 16) {
    if (nu <= 12) return window_dots_n<12, false, NW>(v, S, s_off, nu, N, body);
    if (nu <= 16 || NW == 16) return window_dots_n<16, false, NW>(v, S, s_off, nu, N, body);
    if constexpr (NW >= 32) {
      if (nu <= 20) return window_dots_n<20, LEAN, NW>(v, S, s_off, nu, N, body);
      if (nu <= 24) return window_dots_n<24, LEAN, NW>(v, S, s_off, nu, N, body);
      if (nu <= 28) return window_dots_n<28, LEAN, NW>(v, S, s_off, nu, N, body);
      return window_dots_n<32, LEAN, NW>(v, S, s_off, nu, N, body);
    }
  }
  return 0.0;
}

// Grid of a window-dots kernel: four elements per thread once that still fills
// the GPU with two blocks per SM (the tail of 31 FP64 additions per warp is
// shared by more products), fewer below, and at most kWinBlocksPerSm blocks
// per SM.
inline int window_dots_blocks(const pfk_context* ctx, int64_t N) {
  const int64_t cap = (int64_t)ctx->num_sms * kWinBlocksPerSm, two = (int64_t)ctx->num_sms * 2;
  const int64_t one = (N + kWinThreads - 1) / kWinThreads, four = (N + 4 * kWinThreads - 1) / (4 * kWinThreads);
  const int64_t b = four >= two ? four : (one < two ? one : two);
  return (int)(b < cap ? b : cap);
}

// Persistent single-launch iterations (persistent.cu): eligibility, and one
// cooperative launch of up to `iters` PIPEFCG (pipelined) or FCG iterations.
// FCG passes w, m0, m1, n, Q, Z as null.
constexpr int kPersistentIters = 16;
bool persistent_eligible(const pfk_context* ctx, const pfk_operator* op, const pfk_pc* pc, int method, int naive_like,
                         int64_t N);
cudaError_t launch_persistent(const SolveEnv& env, bool pipelined, int mmax, double* x, double* r, double* u,
                              double* w, double* m0, double* m1, double* n, double* P, double* S, double* Q,
                              double* Z, int iters);

Method* make_pipefcg(bool naive);
Method* make_pipegcr_w();
Method* make_pipefcg_theta();
Method* make_pipegcr();
Method* make_pipefgmres(double sigma);
Method* make_fcg();
Method* make_gcr();
Method* make_fgmres();

// ---------------------------------------------------------------------------
// Scalar phase shared by the CG- and CR-type methods (runs in one thread of the
// last block of the kernel that completed the iteration's reduction)
// ---------------------------------------------------------------------------

// Truncation (Sec. 5): standard nu_i = min(i, nu_max); restart-style
// nu_i = ((i - 1) mod nu_max) + 1.
__device__ __forceinline__ int nu_window(int i, int mmax, int truncation) {
  return truncation == PFK_TRUNC_RESTART ? ((i - 1) % mmax) + 1 : (i < mmax ? i : mmax);
}

__device__ __forceinline__ void push_history(SolveCtl* c, double rho, double rn, double eta, double alpha) {
  if (c->history && c->hist_len < c->hist_cap) {
    double* h = c->history + (size_t)c->hist_len * PFK_HISTORY_FIELDS;
    h[0] = rho; h[1] = rn; h[2] = eta; h[3] = alpha;
  }
  c->hist_len += 1;
}

__device__ __forceinline__ double cgcr_rho(const SolveCtl* ctl, double gamma, double rr) {
  return ctl->norm == PFK_NORM_NATURAL ? sqrt(fabs(gamma)) : sqrt(rr);
}

// Pipeline fill: gamma_0, eta_0 (= delta_0 for Alg. 8, <s_0, s_0> for Alg. 11),
// ||r_0||^2 -> rho_0, target, alpha_0 = gamma_0 / eta_0 and the fill status.
__device__ __forceinline__ void cgcr_fill_scalars(SolveCtl* ctl, double gamma, double eta, double rr) {
  const double rho = cgcr_rho(ctl, gamma, rr);
  if (!ctl->target_set) {
    ctl->rho0 = rho;
    ctl->target = fmax(ctl->rtol * rho, ctl->atol);
    ctl->target_set = 1;
  }
  const double al = eta != 0.0 ? gamma / eta : nan("");
  push_history(ctl, rho, sqrt(rr), eta, al);
  ctl->rho = rho;
  ctl->gamma = gamma;
  ctl->eta = eta;
  ctl->alpha = al;
  ctl->i = 0;
  ctl->nw = 0;
  ctl->eta_ring[0] = eta;
  if (!isfinite(rho)) ctl->status = kNonFinite;
  else if (rho <= ctl->target) ctl->status = kConverged;
  else if (eta <= 0.0) ctl->status = kFillBreakdown;
  else ctl->status = kRun;
}

// Iteration i once its reduction is complete: gamma_i, delta_i, ||r_i||^2 and
// the window dots c[jj] = <v_i, s_k>, k = i - nu_i + jj (v = u for Alg. 8,
// w for Alg. 11).  Convergence test first (as in the listings' order), then
// beta_{i,k} = -c_k / eta_k, eta_i = delta_i - sum_k beta_{i,k}^2 eta_k (k
// ascending), alpha_i = gamma_i / eta_i; eta_i <= 0 is a norm breakdown.
//
// Run by all threads of the (last) block (at least 96): the nu betas (each a
// global load of eta_k and a division) one per thread of warp 0, rho and the
// convergence test by thread 32 and ||r_i|| by thread 64 meanwhile -- a division
// or square root is a chain of FP64 instructions of about a microsecond --, then
// thread 0 accumulates eta_i.  The betas of an iteration that stops here are
// not used.  c: shared or global memory; s_tmp holds 2 * cap + 1 doubles of
// shared memory, cap >= nu.
__device__ __forceinline__ void cgcr_iteration_scalars_block(SolveCtl* ctl, int i, int nu, double gamma, double delta,
                                                             double rr, const double* c, double* s_tmp, int cap) {
  __shared__ double s_rho, s_rnorm;
  int* s_go = (int*)(s_tmp + 2 * cap);
  const int slots = ctl->mmax + 1;
  if ((int)threadIdx.x < nu) {
    const int k = i - nu + (int)threadIdx.x;
    const double ek = ctl->eta_ring[k % slots];
    const double b = -c[threadIdx.x] / ek;
    ctl->beta[threadIdx.x] = b;
    s_tmp[threadIdx.x] = b * b;
    s_tmp[cap + threadIdx.x] = ek;
  } else if (threadIdx.x == 32) {
    const double rho = cgcr_rho(ctl, gamma, rr);
    s_rho = rho;
    ctl->rho = rho;
    s_go[0] = 1;
    if (!isfinite(rho)) { ctl->status = kNonFinite; s_go[0] = 0; }
    else if (rho <= ctl->target) { ctl->status = kConverged; s_go[0] = 0; }
  } else if (threadIdx.x == 64) {
    s_rnorm = sqrt(rr);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const int it = ctl->it + 1;
  ctl->it = it;
  ctl->i = i;
  ctl->gamma = gamma;
  ctl->delta = delta;
  if (!s_go[0]) {
    push_history(ctl, s_rho, s_rnorm, nan(""), nan(""));
    return;
  }
  double sumb = 0.0;
  for (int jj = 0; jj < nu; ++jj) sumb = fma(s_tmp[jj], s_tmp[cap + jj], sumb);
  const double eta = delta - sumb;
  const double al = eta != 0.0 ? gamma / eta : nan("");
  ctl->eta = eta;
  ctl->alpha = al;
  ctl->nw = nu;
  ctl->eta_ring[i % slots] = eta;
  push_history(ctl, s_rho, s_rnorm, eta, al);
  if (eta <= 0.0) { ctl->status = kBreakdown; return; }
  if (it >= ctl->maxit) { ctl->status = kMaxit; return; }
}

}  // namespace pfk
