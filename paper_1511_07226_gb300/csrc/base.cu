// The non-pipelined flexible methods on one GPU, as comparison baselines:
// FCG (Alg. 2), GCR (Alg. 9) and FGMRES (Alg. 13, classical Gram-Schmidt as
// printed).  Their reductions block: each iteration has two reduction phases
// whose results the very next kernel needs (FCG: gamma and the betas, then
// eta; GCR: the betas, then gamma and eta; FGMRES: the Gram-Schmidt
// coefficients, then the norm).  On one GPU "blocking" means a kernel
// boundary plus a last-block combine, with no host round trip.
#include "pfk_internal.cuh"
#include "solver.cuh"
#include "stencil.cuh"
#include "stencil_flat.cuh"

#include <cmath>

namespace pfk {

// Window dots with a pinned order (SolveEnv::pcc): a warp's 32 elements one after
// the other, lane j holding slot j, the vectors transposed through shared memory.
constexpr int kPinThreads = 128;
constexpr int kPinBlocksPerSm = 6;
constexpr int kPinStride = kPinThreads + 1;
static_assert(kWinBlocksPerSm <= kMaxBlocksPerSm && kPinBlocksPerSm <= kMaxBlocksPerSm,
              "partials are sized for kMaxBlocksPerSm blocks per SM");

// A CSR operator (stencil operators take the flat rows, or the tiled walk for
// sums in a pinned order).
struct CsrView {
  const int32_t* rowptr;
  const int32_t* colidx;
  const double* vals;
};

static CsrView csr_of(const pfk_operator* op) {
  CsrView A;
  A.rowptr = op->rowptr; A.colidx = op->colidx; A.vals = op->vals;
  return A;
}

// (A m)_r of a CSR operator.
__device__ __forceinline__ double base_row(const CsrView& A, const double* __restrict__ m, int64_t r) {
  double acc = 0.0;
  for (int32_t p = A.rowptr[r]; p < A.rowptr[r + 1]; ++p) acc = fma(A.vals[p], m[A.colidx[p]], acc);
  return acc;
}

// ---------------------------------------------------------------------------
// Building blocks
// ---------------------------------------------------------------------------

// x_i = x_{i-1} + alpha p_{i-1}, r_i = r_{i-1} - alpha s_{i-1} (slot of i-1).
__global__ void __launch_bounds__(kThreads) base_advance(double* __restrict__ x, double* __restrict__ r,
                                                         const double* __restrict__ P, const double* __restrict__ S,
                                                         int64_t N, const SolveCtl* ctl) {
  if (ctl->status != kRun) return;
  const double alpha = ctl->alpha;
  const size_t off = (size_t)(ctl->i % (ctl->mmax + 1)) * (size_t)N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
    x[e] = fma(alpha, P[off + e], x[e]);
    r[e] = fma(-alpha, S[off + e], r[e]);
  }
}

template <int NW, typename F>
__device__ __forceinline__ double window_dots_pinned(const double* __restrict__ v, const double* __restrict__ S,
                                                     const size_t* s_off, int nu, int64_t N, F&& body) {
  __shared__ double s_sk[NW * kPinStride];
  __shared__ double s_v[kPinThreads];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* my = s_sk + threadIdx.x;
  const double* wv = s_v + warp * 32;
  const double* lrow = s_sk + lane * kPinStride + warp * 32;
  double gw = 0.0;
  for (int64_t base = (int64_t)blockIdx.x * kPinThreads; base < N; base += (int64_t)gridDim.x * kPinThreads) {
    const int64_t e = base + threadIdx.x;
    double vv = 0.0;
    if (e < N) {
      vv = v[e];
      body(e, vv);
    }
#pragma unroll
    for (int j = 0; j < NW; ++j)
      if (j < nu) my[j * kPinStride] = e < N ? S[s_off[j] + e] : 0.0;
    s_v[threadIdx.x] = vv;
    __syncwarp();
    if (lane < nu) {
      double c = gw;
#pragma unroll 8
      for (int t = 0; t < 32; ++t) c = fma(wv[t], lrow[t], c);
      gw = c;
    }
    __syncwarp();
  }
  return gw;
}

// Dots of a vector v with r (<v, r>), of r with itself, and with the stored
// s_k of the window W_i.  Mode FCG: v = u = B(r_i): convergence test on gamma_i =
// <u_i, r_i>, then the betas.  Mode GCR: v = A u_i: the betas only.
enum { kDotsFcg = 0, kDotsGcr = 1 };

// The scalar step after the dots (all threads of the last block): c the
// window's, gamma and rr (FCG) <v, r> and <r, r>.
__device__ __forceinline__ void base_window_scalars(SolveCtl* ctl, int i, int nu, int slots, int mode,
                                                    const double* c, double gamma, double rr) {
  // beta_{i,k} = -<v, s_k> / eta_k, one division per thread (a serial loop of
  // nu divisions in one thread took 25-30 us at nu = 30); not used when the
  // iteration stops here
  if ((int)threadIdx.x < nu)
    ctl->beta[threadIdx.x] = -c[threadIdx.x] / ctl->eta_ring[(i - nu + (int)threadIdx.x) % slots];
  if (threadIdx.x != 0) return;
  ctl->nw = nu;
  if (mode == kDotsFcg) {
    // Alg. 2: gamma_i = <u_i, r_i>, convergence
    ctl->it += 1;
    ctl->gamma = gamma;
    const double rho = cgcr_rho(ctl, gamma, rr);
    ctl->rho = rho;
    push_history(ctl, rho, sqrt(rr), nan(""), nan(""));
    if (!isfinite(rho)) { ctl->status = kNonFinite; return; }
    if (rho <= ctl->target) { ctl->status = kConverged; ctl->i = i; return; }
  }
}

template <int NW>
__global__ void __launch_bounds__(kWinThreads, kWinBlocksPerSm) base_window_dots(const double* __restrict__ v,
                                                                                 const double* __restrict__ r,
                                                                                 const double* __restrict__ S,
                                                                                 int64_t N, SolveCtl* ctl,
                                                                                 double* partials, int mode) {
  if (ctl->status != kRun) return;
  constexpr int ND = NW + 2;
  constexpr int NWARPS = kWinThreads / 32;
  __shared__ size_t s_off[NW];
  __shared__ double s_red[NWARPS * ND];
  __shared__ double s_sum[ND];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = ctl->i + 1;
  const int nu = nu_window(i, ctl->mmax, ctl->truncation);
  const int slots = ctl->mmax + 1;
  const int ng = mode == kDotsFcg ? 2 : 0;   // <v, r> and <r, r> after the window's dots
  if (threadIdx.x < nu) s_off[threadIdx.x] = (size_t)((i - nu + (int)threadIdx.x) % slots) * (size_t)N;
  __syncthreads();
  double g0 = 0.0, g1 = 0.0;
  const double tot = window_dots<NW>(v, S, s_off, nu, N, [&](int64_t e, double ve) {
    if (ng) {
      const double re = __ldg(&r[e]);
      g0 = fma(ve, re, g0);
      g1 = fma(re, re, g1);
    }
  });
  {
    const int nd = nu + ng;
    const int j = lane / (32 / NW);   // the slot whose sum the lane holds
    if (lane % (32 / NW) == 0 && j < nu) s_red[warp * nd + j] = tot;
    if (ng) {
      double g[2] = {g0, g1};
      const double w = warp_sum_transposed<2>(g);
      if (lane % 16 == 0) s_red[warp * nd + nu + lane / 16] = w;
    }
    __syncthreads();
  }
  if (!combine_block_partials_2l(s_red, nu + ng, partials, ND, &ctl->counter, ctl->gcounter, s_sum)) return;
  base_window_scalars(ctl, i, nu, slots, mode, s_sum, s_sum[nu], s_sum[nu + 1]);
}

// The same with the pinned order.
template <int NW>
__global__ void __launch_bounds__(kPinThreads, kPinBlocksPerSm) base_window_dots_pinned(
    const double* __restrict__ v, const double* __restrict__ r, const double* __restrict__ S, int64_t N,
    SolveCtl* ctl, double* partials, int mode) {
  if (ctl->status != kRun) return;
  constexpr int ND = NW + 2;
  constexpr int NWARPS = kPinThreads / 32;
  __shared__ size_t s_off[NW];
  __shared__ double s_red[NWARPS * ND];
  __shared__ double s_sum[ND];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = ctl->i + 1;
  const int nu = nu_window(i, ctl->mmax, ctl->truncation);
  const int slots = ctl->mmax + 1;
  if (threadIdx.x < nu) s_off[threadIdx.x] = (size_t)((i - nu + (int)threadIdx.x) % slots) * (size_t)N;
  __syncthreads();
  double g0 = 0.0, g1 = 0.0;
  const double gw = window_dots_pinned<NW>(v, S, s_off, nu, N, [&](int64_t e, double ve) {
    const double re = r[e];
    g0 = fma(ve, re, g0);
    g1 = fma(re, re, g1);
  });
  const double w0 = warp_sum(g0), w1 = warp_sum(g1);
  const int nd = nu + 2;
  if (lane == 0) {
    s_red[warp * nd + 0] = w0;
    s_red[warp * nd + 1] = w1;
  }
  if (lane < nu) s_red[warp * nd + 2 + lane] = gw;
  __syncthreads();
  if (!combine_block_partials_2l(s_red, nd, partials, ND, &ctl->counter, ctl->gcounter, s_sum)) return;
  base_window_scalars(ctl, i, nu, slots, mode, s_sum + 2, s_sum[0], s_sum[1]);
}

// p_i = u + sum_k beta_{i,k} p_k over W_i, into ring slot i.
template <int NW>
__global__ void __launch_bounds__(kThreads, 3) base_maxpy(const double* __restrict__ u, double* __restrict__ P,
                                                           int64_t N, const SolveCtl* ctl) {
  if (ctl->status != kRun) return;
  __shared__ double s_b[NW];
  __shared__ size_t s_off[NW];
  const int i = ctl->i + 1;
  const int nu = ctl->nw;
  const int slots = ctl->mmax + 1;
  if (threadIdx.x < nu) {
    s_b[threadIdx.x] = ctl->beta[threadIdx.x];
    s_off[threadIdx.x] = (size_t)((i - nu + (int)threadIdx.x) % slots) * (size_t)N;
  }
  __syncthreads();
  const size_t out = (size_t)(i % slots) * (size_t)N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
    double p = u[e];
#pragma unroll 4
    for (int j = 0; j < nu; ++j) p = fma(s_b[j], P[s_off[j] + e], p);
    P[out + e] = p;
  }
}

// s = A p for p in ring slot 0 (fills) or slot i of the current iteration,
// with the dots its scalar step reads: <p, s> (FCG eta), <p, s>, <p, r>,
// <r, r> (FCG fill) or <s, s>, <r, s>, <r, r> (GCR fill and final); the last
// block runs the scalar step.  Only these products are formed: with all five
// dots of <p, r>, <p, s>, <r, s>, <s, s>, <r, r> the FCG walk issued 12 FP64
// instructions per cell instead of 8.
enum { kApplyFcgFill = 0, kApplyFcgEta = 1, kApplyGcrFill = 2, kApplyGcrFinal = 3 };

template <int MODE>
struct ApplyDots {
  static constexpr bool fcg = MODE == kApplyFcgFill || MODE == kApplyFcgEta;
  static constexpr int nd = MODE == kApplyFcgEta ? 1 : 3;
  static __device__ __forceinline__ void add(double (&acc)[nd], double pv, double sv, double rv) {
    acc[0] = fma(fcg ? pv : sv, sv, acc[0]);
    if constexpr (nd == 3) {
      acc[1] = fma(rv, fcg ? pv : sv, acc[1]);
      acc[2] = fma(rv, rv, acc[2]);
    }
  }
};

// The scalar step after s = A p and its dots (last block, one thread): q0 =
// <p, s> or <s, s>, q1 = <p, r> or <r, s>, rr = <r, r>.
template <int MODE>
__device__ __forceinline__ void base_apply_scalars(SolveCtl* ctl, int i, int slots, double q0, double q1, double rr) {
  if (MODE == kApplyFcgFill || MODE == kApplyGcrFill) {
    // FCG: gamma_0 = <u_0, r_0>, eta_0 = <p_0, s_0>; GCR: gamma_0 = <r_0, s_0>, eta_0 = <s_0, s_0>
    cgcr_fill_scalars(ctl, q1, q0, rr);
    return;
  }
  if (MODE == kApplyFcgEta) {
    // Alg. 2: eta_i = <p_i, s_i>, alpha_i = gamma_i / eta_i
    const double eta = q0;
    const double al = eta != 0.0 ? ctl->gamma / eta : nan("");
    ctl->i = i;
    ctl->eta = eta;
    ctl->alpha = al;
    ctl->eta_ring[i % slots] = eta;
    if (ctl->history && ctl->hist_len - 1 < ctl->hist_cap && ctl->hist_len >= 1) {
      ctl->history[(size_t)(ctl->hist_len - 1) * PFK_HISTORY_FIELDS + 2] = eta;
      ctl->history[(size_t)(ctl->hist_len - 1) * PFK_HISTORY_FIELDS + 3] = al;
    }
    if (eta <= 0.0) { ctl->status = kBreakdown; return; }
    if (ctl->it >= ctl->maxit) { ctl->status = kMaxit; return; }
    return;
  }
  // Alg. 9 (standard reading): gamma_i = <r_i, s_i>, eta_i = <s_i, s_i>; convergence,
  // then alpha_i = gamma_i / eta_i
  const double ss = q0, rs = q1;
  ctl->it += 1;
  ctl->i = i;
  ctl->gamma = rs;
  const double rho = cgcr_rho(ctl, rs, rr);
  ctl->rho = rho;
  const double al = ss != 0.0 ? rs / ss : nan("");
  push_history(ctl, rho, sqrt(rr), ss, al);
  if (!isfinite(rho)) { ctl->status = kNonFinite; return; }
  if (rho <= ctl->target) { ctl->status = kConverged; return; }
  ctl->eta = ss;
  ctl->alpha = al;
  ctl->eta_ring[i % slots] = ss;
  if (ss <= 0.0) { ctl->status = kBreakdown; return; }
  if (ctl->it >= ctl->maxit) { ctl->status = kMaxit; return; }
}

// CSR operators: one row per thread.
template <int MODE>
__global__ void __launch_bounds__(kThreads) base_apply_dots(CsrView A, double* __restrict__ P,
                                                            double* __restrict__ S, const double* __restrict__ r,
                                                            int64_t N, SolveCtl* ctl, double* partials) {
  if (ctl->status != kRun) return;
  using D = ApplyDots<MODE>;
  const bool fill = (MODE == kApplyFcgFill || MODE == kApplyGcrFill);
  const int i = fill ? 0 : ctl->i + 1;
  const int slots = ctl->mmax + 1;
  const size_t off = (size_t)(i % slots) * (size_t)N;
  const double* p = P + off;
  double* s = S + off;
  double acc[D::nd] = {};
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
    const double sv = base_row(A, p, e);
    s[e] = sv;
    D::add(acc, p[e], sv, D::nd == 3 ? r[e] : 0.0);
  }
  __shared__ double s_sum[3];
  if (!reduce_last_block_wide<D::nd>(acc, partials, &ctl->counter, s_sum)) return;
  if (threadIdx.x != 0) return;
  base_apply_scalars<MODE>(ctl, i, slots, s_sum[0], s_sum[1], s_sum[2]);
}

// Stencil operators, pinned order: the same step on the tiled z-marching walk (s =
// A p and the dots in its epilogue, r prefetched one plane ahead where it is read).
template <int MODE>
struct BaseApplyEpi {
  using D = ApplyDots<MODE>;
  double* __restrict__ s;
  const double* __restrict__ r;
  double acc[D::nd];
  struct Pre {
    double r;
  };
  __device__ __forceinline__ Pre pre(int64_t c) const { return Pre{D::nd == 3 ? r[c] : 0.0}; }
  __device__ __forceinline__ void operator()(int64_t c, double sv, double pv, const Pre& p) {
    s[c] = sv;
    D::add(acc, pv, sv, p.r);
  }
};

// Planes per work unit, and with them the order of the sums, are chosen for this
// many resident blocks per SM, not for what a build's registers allow.
constexpr int kWalkBlocksPerSm = 2;

template <bool ADV, int MODE>
__global__ void __launch_bounds__(kTileThreads) base_apply_dots_walk(TiledStencil<double, double> T,
                                                                     double* __restrict__ P, double* __restrict__ S,
                                                                     const double* __restrict__ r, int64_t N,
                                                                     SolveCtl* ctl, double* partials) {
  if (ctl->status != kRun) return;
  constexpr int ND = ApplyDots<MODE>::nd;
  const bool fill = (MODE == kApplyFcgFill || MODE == kApplyGcrFill);
  const int i = fill ? 0 : ctl->i + 1;
  const int slots = ctl->mmax + 1;
  const size_t off = (size_t)(i % slots) * (size_t)N;
  BaseApplyEpi<MODE> e{S + off, r, {}};
  tiled_stencil_walk<double, double, ADV, 1>(T, P + off, e);
  __shared__ double s_sum[3];
  if (!reduce_last_block_wide<ND>(e.acc, partials, &ctl->counter, s_sum)) return;
  if (threadIdx.x != 0) return;
  base_apply_scalars<MODE>(ctl, i, slots, s_sum[0], s_sum[1], s_sum[2]);
}

// The same on the flat rows, in their order (ncu, 101x97x93, FCG's eta: 44.8 -> 20.4 us,
// of which the dots no longer formed are a third).
template <bool ADV, int MODE, typename I>
__global__ void __launch_bounds__(kThreads) base_apply_dots_flat(FlatStencilT<I> A, double* __restrict__ P,
                                                                 double* __restrict__ S, const double* __restrict__ r,
                                                                 int64_t N, SolveCtl* ctl, double* partials) {
  if (ctl->status != kRun) return;
  constexpr int ND = ApplyDots<MODE>::nd;
  const bool fill = (MODE == kApplyFcgFill || MODE == kApplyGcrFill);
  const int i = fill ? 0 : ctl->i + 1;
  const int slots = ctl->mmax + 1;
  const size_t off = (size_t)(i % slots) * (size_t)N;
  BaseApplyEpi<MODE> e{S + off, r, {}};
  const double* p = P + off;
  FLAT_CELLS(I, c, A.n) {
    const auto pre = e.pre(c);
    double pv;
    const double sv = flat_row<ADV>(A, p, c, pv);
    e(c, sv, pv, pre);
  }
  __shared__ double s_sum[3];
  if (!reduce_last_block_fast<ND, true>(e.acc, partials, &ctl->counter, s_sum)) return;
  if (threadIdx.x != 0) return;
  base_apply_scalars<MODE>(ctl, i, slots, s_sum[0], s_sum[1], s_sum[2]);
}

static int base_template(int mmax) { return mmax <= 8 ? 8 : mmax <= 16 ? 16 : 32; }

static int pinned_dots_blocks(const SolveEnv& env) {
  const int64_t need = (env.N + kPinThreads - 1) / kPinThreads, cap = (int64_t)env.ctx->num_sms * kPinBlocksPerSm;
  return (int)(need < cap ? need : cap);
}

static cudaError_t launch_window_dots(const SolveEnv& env, int tmpl, const double* v, const double* r,
                                      const double* S, int mode) {
  if (env.pcc.pinned) {
    const int blocks = pinned_dots_blocks(env);
    if (!env.partials_fit_2l(blocks, tmpl + 2)) return cudaErrorInvalidValue;
    switch (tmpl) {
      case 8: base_window_dots_pinned<8><<<blocks, kPinThreads, 0, env.st>>>(v, r, S, env.N, env.ctl, env.partials, mode); break;
      case 16: base_window_dots_pinned<16><<<blocks, kPinThreads, 0, env.st>>>(v, r, S, env.N, env.ctl, env.partials, mode); break;
      default: base_window_dots_pinned<32><<<blocks, kPinThreads, 0, env.st>>>(v, r, S, env.N, env.ctl, env.partials, mode); break;
    }
    return cudaGetLastError();
  }
  const int blocks = window_dots_blocks(env.ctx, env.N);
  if (!env.partials_fit_2l(blocks, tmpl + 2)) return cudaErrorInvalidValue;
  switch (tmpl) {
    case 8: base_window_dots<8><<<blocks, kWinThreads, 0, env.st>>>(v, r, S, env.N, env.ctl, env.partials, mode); break;
    case 16: base_window_dots<16><<<blocks, kWinThreads, 0, env.st>>>(v, r, S, env.N, env.ctl, env.partials, mode); break;
    default: base_window_dots<32><<<blocks, kWinThreads, 0, env.st>>>(v, r, S, env.N, env.ctl, env.partials, mode); break;
  }
  return cudaGetLastError();
}

static cudaError_t launch_maxpy(const SolveEnv& env, int tmpl, const double* u, double* P) {
  const int blocks = stream_blocks(env.ctx, env.N, 4);
  switch (tmpl) {
    case 8: base_maxpy<8><<<blocks, kThreads, 0, env.st>>>(u, P, env.N, env.ctl); break;
    case 16: base_maxpy<16><<<blocks, kThreads, 0, env.st>>>(u, P, env.N, env.ctl); break;
    default: base_maxpy<32><<<blocks, kThreads, 0, env.st>>>(u, P, env.N, env.ctl); break;
  }
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_apply_dots(const SolveEnv& env, double* P, double* S, const double* r) {
  const pfk_operator* op = env.op;
  constexpr int ND = ApplyDots<MODE>::nd;
  if (!op->rowptr && !env.pcc.pinned) {
    const int blocks = stream_blocks(env.ctx, env.N, 4);
    if (!env.partials_fit(blocks, ND)) return cudaErrorInvalidValue;
    with_flat_stencil(op, [&](const auto& A, auto adv) {
      base_apply_dots_flat<adv.value, MODE><<<blocks, kThreads, 0, env.st>>>(A, P, S, r, env.N, env.ctl,
                                                                             env.partials);
    });
    return cudaGetLastError();
  }
  if (!op->rowptr) {
    TiledStencil<double, double> T;
    const bool adv = op->adv[0] != 0.0 || op->adv[1] != 0.0 || op->adv[2] != 0.0;
    const int slots = kWalkBlocksPerSm * env.ctx->num_sms;
    const int units = tiled_stencil_setup<double, double>(T, op, op->d, op->kx, op->ky, op->kz, slots);
    const int64_t cap = env.partials_cap / 5;   // (part of the order: blocks take units u, u + blocks, ...)
    const int blocks = (int)(units < cap ? units : cap);
    if (adv) base_apply_dots_walk<true, MODE><<<blocks, kTileThreads, 0, env.st>>>(T, P, S, r, env.N, env.ctl, env.partials);
    else base_apply_dots_walk<false, MODE><<<blocks, kTileThreads, 0, env.st>>>(T, P, S, r, env.N, env.ctl, env.partials);
    return cudaGetLastError();
  }
  const int blocks = stream_blocks(env.ctx, env.N, 2);
  if (!env.partials_fit(blocks, ND)) return cudaErrorInvalidValue;
  base_apply_dots<MODE><<<blocks, kThreads, 0, env.st>>>(csr_of(env.op), P, S, r, env.N, env.ctl, env.partials);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FCG (Alg. 2)
// ---------------------------------------------------------------------------

class Fcg : public Method {
 public:
  int64_t workspace_doubles(int64_t N, int mmax) const override { return 3 * N + 2 * (int64_t)(mmax + 1) * N; }
  void bind(double* ws, int64_t N, int mmax) override {
    N_ = N; mmax_ = mmax;
    r_ = ws; u_ = r_ + N; tmp_ = u_ + N;
    P_ = tmp_ + N; S_ = P_ + (mmax + 1) * N;
  }
  double* scratch() override { return tmp_; }
  bool blocking() const override { return true; }
  int iterations_per_step() const override { return persistent_ ? kPersistentIters : 1; }
  bool configure(const pfk_context* ctx, const pfk_operator* op, const pfk_pc* pc, int64_t N, int mode) override {
    persistent_ = mode != 1 && persistent_eligible(ctx, op, pc, PFK_FCG, 0, N);
    return persistent_;
  }
  cudaError_t fill(const SolveEnv& env, const double* b, double* x) override {
    cudaError_t e;
    if ((e = op_apply(env.op, x, r_, b, nullptr, env.st)) != cudaSuccess) return e;   // r_0 = b - A x_0
    if ((e = env.pc_apply(r_, P_, nullptr, nullptr)) != cudaSuccess) return e;       // p_0 = u_0 = B(r_0)
    return launch_apply_dots<kApplyFcgFill>(env, P_, S_, r_);                          // s_0 = A p_0, gamma_0, eta_0
  }
  cudaError_t iteration(const SolveEnv& env, double* x) override {
    if (persistent_) {
      cudaError_t e = env.mark_pass(0);
      if (e != cudaSuccess) return e;
      e = launch_persistent(env, false, mmax_, x, r_, u_, nullptr, nullptr, nullptr, nullptr, P_, S_, nullptr,
                            nullptr, kPersistentIters);
      if (e != cudaSuccess) return e;
      return env.mark_pass(1);
    }
    const int* status = &env.ctl->status;
    const int tmpl = base_template(mmax_);
    cudaError_t e;
    base_advance<<<stream_blocks(env.ctx, N_, 8), kThreads, 0, env.st>>>(x, r_, P_, S_, N_, env.ctl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = env.pc_apply(r_, u_, nullptr, status)) != cudaSuccess) return e;         // u_i = B(r_i)
    if ((e = env.mark_pass(0)) != cudaSuccess) return e;
    if ((e = launch_window_dots(env, tmpl, u_, r_, S_, kDotsFcg)) != cudaSuccess) return e;   // gamma_i, betas
    if ((e = launch_maxpy(env, tmpl, u_, P_)) != cudaSuccess) return e;                // p_i
    if ((e = launch_apply_dots<kApplyFcgEta>(env, P_, S_, r_)) != cudaSuccess) return e;      // s_i, eta_i, alpha_i
    return env.mark_pass(1);
  }

 private:
  int64_t N_ = 0;
  int mmax_ = 0;
  bool persistent_ = false;
  double *r_ = nullptr, *u_ = nullptr, *tmp_ = nullptr, *P_ = nullptr, *S_ = nullptr;
};

// ---------------------------------------------------------------------------
// GCR (Alg. 9)
// ---------------------------------------------------------------------------

class Gcr : public Method {
 public:
  int64_t workspace_doubles(int64_t N, int mmax) const override { return 4 * N + 2 * (int64_t)(mmax + 1) * N; }
  void bind(double* ws, int64_t N, int mmax) override {
    N_ = N; mmax_ = mmax;
    r_ = ws; u_ = r_ + N; au_ = u_ + N; tmp_ = au_ + N;
    P_ = tmp_ + N; S_ = P_ + (mmax + 1) * N;
  }
  double* scratch() override { return tmp_; }
  bool blocking() const override { return true; }
  cudaError_t fill(const SolveEnv& env, const double* b, double* x) override {
    cudaError_t e;
    if ((e = op_apply(env.op, x, r_, b, nullptr, env.st)) != cudaSuccess) return e;   // r_0
    if ((e = env.pc_apply(r_, P_, nullptr, nullptr)) != cudaSuccess) return e;       // p_0 = u_0 = B(r_0)
    return launch_apply_dots<kApplyGcrFill>(env, P_, S_, r_);                          // s_0, gamma_0, eta_0
  }
  cudaError_t iteration(const SolveEnv& env, double* x) override {
    const int* status = &env.ctl->status;
    const int tmpl = base_template(mmax_);
    cudaError_t e;
    base_advance<<<stream_blocks(env.ctx, N_, 8), kThreads, 0, env.st>>>(x, r_, P_, S_, N_, env.ctl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = env.pc_apply(r_, u_, nullptr, status)) != cudaSuccess) return e;         // u_i = B(r_i)
    if ((e = env.mark_pass(0)) != cudaSuccess) return e;
    if ((e = op_apply(env.op, u_, au_, nullptr, status, env.st)) != cudaSuccess) return e;   // A u_i
    if ((e = launch_window_dots(env, tmpl, au_, r_, S_, kDotsGcr)) != cudaSuccess) return e;  // betas
    if ((e = launch_maxpy(env, tmpl, u_, P_)) != cudaSuccess) return e;                // p_i
    if ((e = launch_apply_dots<kApplyGcrFinal>(env, P_, S_, r_)) != cudaSuccess) return e;    // s_i, gamma, eta
    return env.mark_pass(1);
  }

 private:
  int64_t N_ = 0;
  int mmax_ = 0;
  double *r_ = nullptr, *u_ = nullptr, *au_ = nullptr, *tmp_ = nullptr, *P_ = nullptr, *S_ = nullptr;
};

// ---------------------------------------------------------------------------
// FGMRES (Alg. 13)
// ---------------------------------------------------------------------------

constexpr int kGm = PFK_MAX_MMAX;

struct FgState {
  double H[(kGm + 1) * kGm];
  double R[(kGm + 1) * kGm];
  double cs[kGm], sn[kGm];
  double g[kGm + 1];
  double y[kGm];
  double inv;
  int k;        // column being formed
  int ncols;
};

// beta = ||r_0||, convergence, g = beta e_0.
__global__ void __launch_bounds__(kThreads) fgb_fill_norm(const double* __restrict__ r, int64_t N, SolveCtl* ctl,
                                                          FgState* gs, double* partials) {
  double acc[1] = {0.0};
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x)
    acc[0] = fma(r[e], r[e], acc[0]);
  __shared__ double s_sum[1];
  if (!reduce_last_block_fast<1>(acc, partials, &ctl->counter, s_sum)) return;
  if (threadIdx.x != 0) return;
  const double beta = sqrt(s_sum[0]);
  if (!ctl->target_set) {
    ctl->rho0 = beta;
    ctl->target = fmax(ctl->rtol * beta, ctl->atol);
    ctl->target_set = 1;
  }
  push_history(ctl, beta, beta, nan(""), nan(""));
  ctl->rho = beta;
  ctl->i = 0;
  gs->g[0] = beta;
  gs->k = 0;
  gs->ncols = 0;
  gs->inv = beta != 0.0 ? 1.0 / beta : 0.0;
  if (!isfinite(beta)) ctl->status = kNonFinite;
  else if (beta <= ctl->target) ctl->status = kConverged;
  else if (ctl->it >= ctl->maxit) ctl->status = kMaxit;
  else ctl->status = kRun;
}

// slot k of P (k = gs->k) scaled by gs->inv in place, and copied to `cur`.
__global__ void __launch_bounds__(kThreads) fgb_scale(const double* __restrict__ src, double* __restrict__ P,
                                                      double* __restrict__ cur, int64_t N, const FgState* gs,
                                                      const int* status) {
  if (*status != kRun) return;
  const double inv = gs->inv;
  const size_t off = (size_t)gs->k * (size_t)N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
    const double v = (src ? src[e] : P[off + e]) * inv;
    P[off + e] = v;
    cur[e] = v;
  }
}

// z = A u_k, and u_k stored in slot k of U (CSR operators).
__global__ void __launch_bounds__(kThreads) fgb_apply_store(CsrView A, const double* __restrict__ ucur,
                                                            double* __restrict__ U, double* __restrict__ z, int64_t N,
                                                            const FgState* gs, const int* status) {
  if (*status != kRun) return;
  const size_t off = (size_t)gs->k * (size_t)N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
    z[e] = base_row(A, ucur, e);
    U[off + e] = ucur[e];
  }
}

// The same for stencil operators.
template <bool ADV, typename I>
__global__ void __launch_bounds__(kThreads) fgb_apply_store_flat(FlatStencilT<I> A, const double* __restrict__ ucur,
                                                                 double* __restrict__ U, double* __restrict__ z,
                                                                 int64_t N, const FgState* gs, const int* status) {
  if (*status != kRun) return;
  double* u = U + (size_t)gs->k * (size_t)N;
  FLAT_CELLS(I, c, A.n) {
    double uv;
    z[c] = flat_row<ADV>(A, ucur, c, uv);
    u[c] = uv;
  }
}

static cudaError_t launch_apply_store(const SolveEnv& env, const double* ucur, double* U, double* z,
                                      const FgState* gs, const int* status) {
  const pfk_operator* op = env.op;
  const int blocks = stream_blocks(env.ctx, env.N, 8);
  if (op->rowptr) {
    fgb_apply_store<<<blocks, kThreads, 0, env.st>>>(csr_of(op), ucur, U, z, env.N, gs, status);
  } else {
    with_flat_stencil(op, [&](const auto& A, auto adv) {
      fgb_apply_store_flat<adv.value><<<blocks, kThreads, 0, env.st>>>(A, ucur, U, z, env.N, gs, status);
    });
  }
  return cudaGetLastError();
}

// Classical Gram-Schmidt coefficients h_{j,k} = <p_j, z_k>, j <= k (window_dots).
template <int NW>
__global__ void __launch_bounds__(kWinThreads, kWinBlocksPerSm) fgb_dots(const double* __restrict__ z,
                                                                         const double* __restrict__ P, int64_t N,
                                                                         SolveCtl* ctl, FgState* gs,
                                                                         double* partials) {
  if (ctl->status != kRun) return;
  constexpr int ND = NW;
  constexpr int NWARPS = kWinThreads / 32;
  __shared__ size_t s_off[NW];
  __shared__ double s_red[NWARPS * ND];
  __shared__ double s_sum[ND];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nk = gs->k + 1;           // p_0 .. p_k
  if (threadIdx.x < nk) s_off[threadIdx.x] = (size_t)threadIdx.x * (size_t)N;
  __syncthreads();
  const double tot = window_dots<NW>(z, P, s_off, nk, N, [](int64_t, double) {});
  const int j = lane / (32 / NW);   // the slot whose sum the lane holds
  if (lane % (32 / NW) == 0 && j < nk) s_red[warp * nk + j] = tot;
  __syncthreads();
  if (!combine_block_partials_2l(s_red, nk, partials, ND, &ctl->counter, ctl->gcounter, s_sum)) return;
  if ((int)threadIdx.x < nk) gs->H[threadIdx.x * kGm + gs->k] = s_sum[threadIdx.x];
}

template <int NW>
__global__ void __launch_bounds__(kPinThreads, kPinBlocksPerSm) fgb_dots_pinned(const double* __restrict__ z,
                                                                                const double* __restrict__ P,
                                                                                int64_t N, SolveCtl* ctl, FgState* gs,
                                                                                double* partials) {
  if (ctl->status != kRun) return;
  constexpr int NWARPS = kPinThreads / 32;
  __shared__ size_t s_off[NW];
  __shared__ double s_red[NWARPS * NW];
  __shared__ double s_sum[NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nk = gs->k + 1;           // p_0 .. p_k
  if (threadIdx.x < nk) s_off[threadIdx.x] = (size_t)threadIdx.x * (size_t)N;
  __syncthreads();
  const double gw = window_dots_pinned<NW>(z, P, s_off, nk, N, [](int64_t, double) {});
  if (lane < nk) s_red[warp * nk + lane] = gw;
  __syncthreads();
  if (!combine_block_partials_2l(s_red, nk, partials, NW, &ctl->counter, ctl->gcounter, s_sum)) return;
  if ((int)threadIdx.x < nk) gs->H[threadIdx.x * kGm + gs->k] = s_sum[threadIdx.x];
}

template <int NW>
static void launch_fgb_dots(const SolveEnv& env, const double* z, const double* P, FgState* gs, int blocks) {
  if (env.pcc.pinned)
    fgb_dots_pinned<NW><<<blocks, kPinThreads, 0, env.st>>>(z, P, env.N, env.ctl, gs, env.partials);
  else
    fgb_dots<NW><<<blocks, kWinThreads, 0, env.st>>>(z, P, env.N, env.ctl, gs, env.partials);
}

// pbar = z_k - sum_j h_{j,k} p_j into slot k+1, and ||pbar||^2; the last block
// finishes column k: h_{k+1,k}, Givens, estimate, status.
template <int NW>
__global__ void __launch_bounds__(kThreads, 3) fgb_orth(const double* __restrict__ z, double* __restrict__ P,
                                                        int64_t N, SolveCtl* ctl, FgState* gs, int m,
                                                        double* partials) {
  if (ctl->status != kRun) return;
  __shared__ double s_h[NW];
  const int k = gs->k;
  const int nk = k + 1;
  if (threadIdx.x < nk) s_h[threadIdx.x] = gs->H[threadIdx.x * kGm + k];
  __syncthreads();
  const size_t out = (size_t)(k + 1) * (size_t)N;
  double acc[1] = {0.0};
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
    double v = z[e];
#pragma unroll 4
    for (int j = 0; j < nk; ++j) v = fma(-s_h[j], P[(size_t)j * (size_t)N + e], v);
    if (k + 1 < m) P[out + e] = v;
    acc[0] = fma(v, v, acc[0]);
  }
  __shared__ double s_sum[1];
  if (!reduce_last_block_fast<1>(acc, partials, &ctl->counter, s_sum)) return;
  // column k in shared memory: the rotations are loaded and the column stored
  // by the block's threads, thread 0 runs the recurrence
  __shared__ double s_cs[NW], s_sn[NW], s_r[NW + 1];
  if ((int)threadIdx.x < nk) {
    s_r[threadIdx.x] = s_h[threadIdx.x];
    if ((int)threadIdx.x < k) {
      s_cs[threadIdx.x] = gs->cs[threadIdx.x];
      s_sn[threadIdx.x] = gs->sn[threadIdx.x];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double h = sqrt(s_sum[0]);
    gs->H[(k + 1) * kGm + k] = h;
    ctl->it += 1;
    gs->ncols = k + 1;
    ctl->i = k + 1;
    double a = s_r[0];
    for (int j = 0; j < k; ++j) {
      const double b = s_r[j + 1];
      s_r[j] = s_cs[j] * a + s_sn[j] * b;
      a = -s_sn[j] * a + s_cs[j] * b;
    }
    const double rr = hypot(a, h);
    const double c = rr != 0.0 ? a / rr : 1.0, s = rr != 0.0 ? h / rr : 0.0;
    gs->cs[k] = c;
    gs->sn[k] = s;
    s_r[k] = rr;
    gs->R[(k + 1) * kGm + k] = 0.0;
    const double gk = gs->g[k];
    gs->g[k + 1] = -s * gk;
    gs->g[k] = c * gk;
    const double est = fabs(-s * gk);
    ctl->rho = est;
    push_history(ctl, est, nan(""), nan(""), h);
    gs->inv = h != 0.0 ? 1.0 / h : 0.0;
    gs->k = k + 1;
    if (!isfinite(est)) ctl->status = kNonFinite;
    else if (est <= ctl->target || h == 0.0) ctl->status = kConverged;
    else if (k + 1 == m) ctl->status = kCycleEnd;
    else if (ctl->it >= ctl->maxit) ctl->status = kMaxit;
  }
  __syncthreads();
  if ((int)threadIdx.x < nk) gs->R[threadIdx.x * kGm + k] = s_r[threadIdx.x];
}

__global__ void fgb_lsq(FgState* gs) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int n = gs->ncols;
  for (int j = n - 1; j >= 0; --j) {
    double s = gs->g[j];
    for (int l = j + 1; l < n; ++l) s -= gs->R[j * kGm + l] * gs->y[l];
    gs->y[j] = s / gs->R[j * kGm + j];
  }
}

__global__ void __launch_bounds__(kThreads) fgb_update_x(double* __restrict__ x, const double* __restrict__ U,
                                                         int64_t N, const FgState* gs) {
  const int n = gs->ncols;
  if (n == 0) return;
  __shared__ double s_y[kGm];
  if (threadIdx.x < n) s_y[threadIdx.x] = gs->y[threadIdx.x];
  __syncthreads();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
    double v = x[e];
    for (int j = 0; j < n; ++j) v = fma(s_y[j], U[(size_t)j * (size_t)N + e], v);
    x[e] = v;
  }
}

class Fgmres : public Method {
 public:
  int64_t workspace_doubles(int64_t N, int m) const override {
    return state_doubles() + 5 * N + (int64_t)(m + 1) * N + (int64_t)m * N;
  }
  void bind(double* ws, int64_t N, int m) override {
    N_ = N; m_ = m;
    gs_ = (FgState*)ws;
    double* v = ws + state_doubles();
    r_ = v; z_ = r_ + N; pcur_ = z_ + N; ucur_ = pcur_ + N; tmp_ = ucur_ + N;
    P_ = tmp_ + N; U_ = P_ + (int64_t)(m + 1) * N;
  }
  double* scratch() override { return tmp_; }
  bool blocking() const override { return true; }
  int cycle_length() const override { return m_; }
  cudaError_t fill(const SolveEnv& env, const double* b, double* x) override {
    const int* status = &env.ctl->status;
    const int blocks = stream_blocks(env.ctx, N_, 2);
    if (!env.partials_fit(blocks, 1)) return cudaErrorInvalidValue;
    cudaError_t e;
    if ((e = op_apply(env.op, x, r_, b, nullptr, env.st)) != cudaSuccess) return e;        // r_0
    fgb_fill_norm<<<blocks, kThreads, 0, env.st>>>(r_, N_, env.ctl, gs_, env.partials);      // beta
    fgb_scale<<<stream_blocks(env.ctx, N_, 8), kThreads, 0, env.st>>>(r_, P_, pcur_, N_, gs_, status);  // p_0
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = env.pc_apply(pcur_, ucur_, nullptr, status)) != cudaSuccess) return e;       // u_0 = B(p_0)
    return launch_apply_store(env, ucur_, U_, z_, gs_, status);                            // z_0 = A u_0
  }
  cudaError_t iteration(const SolveEnv& env, double* x) override {
    (void)x;
    const int* status = &env.ctl->status;
    const int tmpl = base_template(m_ + 1);
    const int dblocks = env.pcc.pinned ? pinned_dots_blocks(env) : window_dots_blocks(env.ctx, N_);
    const int oblocks = stream_blocks(env.ctx, N_, 2);
    if (!env.partials_fit_2l(dblocks, tmpl) || !env.partials_fit(oblocks, 1)) return cudaErrorInvalidValue;
    cudaError_t e;
    if ((e = env.mark_pass(0)) != cudaSuccess) return e;
    switch (tmpl) {
      case 8:
        launch_fgb_dots<8>(env, z_, P_, gs_, dblocks);
        fgb_orth<8><<<oblocks, kThreads, 0, env.st>>>(z_, P_, N_, env.ctl, gs_, m_, env.partials);
        break;
      case 16:
        launch_fgb_dots<16>(env, z_, P_, gs_, dblocks);
        fgb_orth<16><<<oblocks, kThreads, 0, env.st>>>(z_, P_, N_, env.ctl, gs_, m_, env.partials);
        break;
      default:
        launch_fgb_dots<32>(env, z_, P_, gs_, dblocks);
        fgb_orth<32><<<oblocks, kThreads, 0, env.st>>>(z_, P_, N_, env.ctl, gs_, m_, env.partials);
        break;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = env.mark_pass(1)) != cudaSuccess) return e;
    fgb_scale<<<stream_blocks(env.ctx, N_, 8), kThreads, 0, env.st>>>(nullptr, P_, pcur_, N_, gs_, status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;                              // p_k = pbar / h
    if ((e = env.pc_apply(pcur_, ucur_, nullptr, status)) != cudaSuccess) return e;    // u_k = B(p_k)
    return launch_apply_store(env, ucur_, U_, z_, gs_, status);                          // z_k = A u_k
  }
  cudaError_t end_cycle(const SolveEnv& env, double* x) override {
    fgb_lsq<<<1, 32, 0, env.st>>>(gs_);
    fgb_update_x<<<stream_blocks(env.ctx, N_, 8), kThreads, 0, env.st>>>(x, U_, N_, gs_);
    return cudaGetLastError();
  }

 private:
  static int64_t state_doubles() { return (int64_t)((sizeof(FgState) + 255) / 256 * 256 / sizeof(double)); }
  int64_t N_ = 0;
  int m_ = 0;
  FgState* gs_ = nullptr;
  double *r_ = nullptr, *z_ = nullptr, *pcur_ = nullptr, *ucur_ = nullptr, *tmp_ = nullptr;
  double *P_ = nullptr, *U_ = nullptr;
};

Method* make_fcg() { return new Fcg(); }
Method* make_gcr() { return new Gcr(); }
Method* make_fgmres() { return new Fgmres(); }

}  // namespace pfk
