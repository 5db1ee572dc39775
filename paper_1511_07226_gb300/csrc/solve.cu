// Solve driver: restarts, residual replacement and graph-replayed iterations.
//
// Host logic only (scalars and control); every vector operation is a kernel of
// the method object.  Per solve:
//   1. the pipeline fill is launched kernel by kernel; meanwhile the host records
//      two iterations into a CUDA graph (all scalars live in the device control
//      block, so a graph is valid for every iteration and restart), launches it
//      for the first `graph_iters` iterations, and records the graph of
//      `graph_iters` iterations while the GPU works on those.  Recording and
//      instantiating the long graph before the first launch left the GPU idle
//      for 0.5 ms of every solve (64^3 PIPEGCR: 706 us for a solve of no
//      iterations); launching the first iterations kernel by kernel costs ~7 us
//      per kernel against ~4 us in a graph;
//   2. iteration-graph launches, two batches in flight, with the status words
//      copied back asynchronously after each; iterations after convergence are
//      no-ops, and no batch is launched past maxit;
//   3. on convergence the true residual ||b - A x|| is checked (residual
//      replacement: restart from x with a tightened target when it fails); on a
//      norm breakdown the method restarts from x, flushing the pipeline
//      (Sec. 5: implementations detect norm breakdown and restart).
#include "pfk_internal.cuh"
#include "solver.cuh"

#include <cmath>
#include <cstring>
#include <memory>
#include <vector>

namespace pfk {

cudaError_t SolveEnv::pc_apply(const double* v, double* out, const double* add, const int* status) const {
  if (pc) return pfk::pc_apply(pc, v, out, add, status, st, pcc);
  pfk_pc id;   // identity
  id.ctx = ctx;
  id.op = op;
  id.kind = PFK_PC_NONE;
  return pfk::pc_apply(&id, v, out, add, status, st, pcc);
}

cudaError_t SolveEnv::mark_pass(int which) const {
  cudaEvent_t e = which == 0 ? pass_ev0 : pass_ev1;
  if (!e) return cudaSuccess;
  return cudaEventRecordWithFlags(e, st, cudaEventRecordExternal);
}

__global__ void ctl_restart_kernel(SolveCtl* ctl) {
  ctl->status = kRun;
  ctl->i = 0;
  ctl->nw = 0;
  ctl->counter = 0u;
}

static Method* make_method(int method, double sigma = NAN) {
  switch (method) {
    case PFK_PIPEFCG: return make_pipefcg(false);
    case PFK_PIPEFCG_NAIVE: return make_pipefcg(true);
    case PFK_PIPEGCR_W: return make_pipegcr_w();
    case PFK_PIPEFCG_THETA: return make_pipefcg_theta();
    case PFK_PIPEGCR: return make_pipegcr();
    case PFK_PIPEFGMRES: return make_pipefgmres(sigma);
    case PFK_FCG: return make_fcg();
    case PFK_GCR: return make_gcr();
    case PFK_FGMRES: return make_fgmres();
    default: return nullptr;
  }
}

// Methods usable as the inner solve of a nested preconditioner (device-only
// control: no restarts, no cycle ends).
Method* make_inner_method(int method) {
  switch (method) {
    case PFK_FCG:
    case PFK_PIPEFCG:
    case PFK_PIPEFCG_THETA:
    case PFK_GCR:
    case PFK_PIPEGCR:
    case PFK_PIPEGCR_W: return make_method(method);
    default: return nullptr;
  }
}

bool method_supported(int method) {
  std::unique_ptr<Method> m(make_method(method));
  return m != nullptr;
}

pfk_status solve_workspace_bytes(int method, int mmax, int64_t n, int64_t* bytes) {
  std::unique_ptr<Method> m(make_method(method));
  if (!m) return PFK_ERR_INVALID;
  *bytes = m->workspace_doubles(n, mmax) * (int64_t)sizeof(double);
  return PFK_OK;
}

namespace {

struct Graph {
  cudaGraph_t g = nullptr;
  cudaGraphExec_t x = nullptr;
  int kernels = 0;
  ~Graph() {
    if (x) cudaGraphExecDestroy(x);
    if (g) cudaGraphDestroy(g);
  }
};

// Records what `body` enqueues on cs; instantiates it unless only the number of
// its kernels is wanted.
template <typename F>
cudaError_t capture(cudaStream_t cs, Graph& out, bool instantiate, F&& body) {
  cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  cudaError_t eb = body();
  e = cudaStreamEndCapture(cs, &out.g);
  if (eb != cudaSuccess) return eb;
  if (e != cudaSuccess) return e;
  size_t nn = 0;
  if ((e = cudaGraphGetNodes(out.g, nullptr, &nn)) != cudaSuccess) return e;
  std::vector<cudaGraphNode_t> nodes(nn);
  if (nn && (e = cudaGraphGetNodes(out.g, nodes.data(), &nn)) != cudaSuccess) return e;
  for (auto& n : nodes) {
    cudaGraphNodeType t;
    if (cudaGraphNodeGetType(n, &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) out.kernels++;
  }
  return instantiate ? cudaGraphInstantiate(&out.x, out.g, 0) : cudaSuccess;
}

struct Events {
  std::vector<cudaEvent_t> v;
  ~Events() {
    for (auto e : v)
      if (e) cudaEventDestroy(e);
  }
  cudaError_t make(int n, unsigned flags) {
    v.assign(n, nullptr);
    for (int i = 0; i < n; ++i) {
      cudaError_t e = cudaEventCreateWithFlags(&v[i], flags);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
};

}  // namespace

pfk_status run_solve(pfk_context* ctx, const pfk_operator* op, const pfk_pc* pc, const pfk_solve_params* prm,
                     const double* b, double* x, pfk_solve_info* info) {
  cudaStream_t st = ctx->stream;
  const int64_t N = op->n;
  const int mmax = prm->mmax;
  std::unique_ptr<Method> M(make_method(prm->method, prm->sigma));
  if (!M) {
    set_error(ctx, "method not available");
    return PFK_ERR_INVALID;
  }
  if (prm->persistent < 0 || prm->persistent > 2) {
    set_error(ctx, "persistent must be 0 (auto), 1 (never) or 2 (required)");
    return PFK_ERR_INVALID;
  }
  if (!M->configure(ctx, op, pc, N, prm->persistent) && prm->persistent == 2) {
    set_error(ctx, "the persistent path needs PIPEFCG or FCG, an assembled CSR operator, Jacobi or no "
                   "preconditioner and n <= PFK_PERSISTENT_MAX_N");
    return PFK_ERR_INVALID;
  }
  // ---- workspace: control block | method vectors | partials | scalars | history ----
  // partials: room for any kernel of the solve (at most kMaxBlocksPerSm blocks
  // per SM, at most kPartialStride values per block); launches check it.
  const int64_t wd = M->workspace_doubles(N, mmax);
  // block rows of the largest reduction grid plus the two-level combine's group rows
  const int64_t pd = ((int64_t)ctx->num_sms * kMaxBlocksPerSm + kMaxCombineGroups) * kPartialStride;
  const int64_t sd = 64;
  const int hist_cap = prm->history ? prm->history_capacity : 0;
  const int64_t hd = (int64_t)hist_cap * PFK_HISTORY_FIELDS;
  const size_t ctl_bytes = (sizeof(SolveCtl) + 255) / 256 * 256;
  const size_t need = (size_t)(wd + pd + sd + hd) * sizeof(double) + ctl_bytes + 256;
  if (ctx->ws_bytes < need) {
    if (ctx->ws) cudaFreeAsync(ctx->ws, st);
    ctx->ws = nullptr;
    ctx->ws_bytes = 0;
    cudaError_t e = cudaMallocAsync(&ctx->ws, need, st);
    if (e != cudaSuccess) {
      cudaGetLastError();
      set_error(ctx, "out of device memory for the solve workspace");
      return PFK_ERR_OOM;
    }
    ctx->ws_bytes = need;
  }
  char* base = (char*)ctx->ws;
  SolveCtl* ctl = (SolveCtl*)base;
  double* ws = (double*)(base + ctl_bytes);
  double* partials = ws + wd;
  double* d_out = partials + pd;
  double* hist = hist_cap ? d_out + sd : nullptr;
  M->bind(ws, N, mmax);

  SolveCtl h;
  std::memset(&h, 0, sizeof(h));
  h.status = kRun;
  h.maxit = prm->maxit;
  h.mmax = mmax;
  h.truncation = prm->truncation;
  h.norm = prm->norm;
  h.rtol = prm->rtol;
  h.atol = prm->atol;
  h.history = hist;
  h.hist_cap = hist_cap;
  h.bar_timeout_ns = prm->barrier_timeout_us == 0 ? kBarrierTimeoutNs
                     : prm->barrier_timeout_us < 0 ? 0ll : 1000ll * (long long)prm->barrier_timeout_us;
  PFK_CUDA(ctx, cudaMemcpyAsync(ctl, &h, sizeof(SolveCtl), cudaMemcpyHostToDevice, st));

  SolveEnv env;
  env.ctx = ctx;
  env.op = op;
  env.pc = pc;
  env.st = st;
  env.ctl = ctl;
  env.partials = partials;
  env.partials_cap = pd;
  env.N = N;
  env.pass_ev0 = env.pass_ev1 = nullptr;
  const bool fp64 = !pc || (pc->kind != PFK_PC_BLOCK_UPPER && pc->precision == PFK_FP64);
  env.pcc = PcCall{!(M->blocking() && fp64), h.bar_timeout_ns, &ctx->pinned->pc_gave_up};

  long long kernel_launches = 0;

  SolveCtl* hc = ctx->pinned->status;
  double* h_bb = ctx->pinned->scalars;

  // ---- ||b||: read after the first synchronisation below ----
  PFK_CUDA(ctx, dot_into(ctx, b, b, N, d_out, st));
  kernel_launches += 1;
  PFK_CUDA(ctx, cudaMemcpyAsync(h_bb, d_out, sizeof(double), cudaMemcpyDeviceToHost, st));
  double sigma_used = NAN;
  PFK_CUDA(ctx, M->prepare(env, b, d_out, &sigma_used));
  const bool gmres = M->cycle_length() > 0;

  // ---- graphs: recorded on the library's own stream (the caller's may be the
  // legacy default stream, which cannot be captured), launched on the caller's ----
  const int K = prm->graph_iters > 0 ? prm->graph_iters : 8;
  const bool profile = prm->profile != 0;
  Events pev;
  if (profile) PFK_CUDA(ctx, pev.make(2 * K, cudaEventDefault));
  constexpr int kShort = 2;
  Graph gfill, giter, gshort;   // (gfill: only counted)
  SolveEnv cenv = env;
  cenv.st = ctx->cap_stream;
  auto record = [&](Graph& g, int iters, bool instantiate) -> cudaError_t {
    return capture(cenv.st, g, instantiate, [&]() -> cudaError_t {
      cudaError_t e2 = cudaSuccess;
      for (int q = 0; q < iters && e2 == cudaSuccess; ++q) {
        SolveEnv ienv = cenv;
        if (profile) {
          ienv.pass_ev0 = pev.v[2 * q];
          ienv.pass_ev1 = pev.v[2 * q + 1];
        }
        e2 = M->iteration(ienv, x);
      }
      return e2;
    });
  };
  auto fill = [&](const SolveEnv& fenv) -> cudaError_t {
    ctl_restart_kernel<<<1, 1, 0, fenv.st>>>(ctl);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : M->fill(fenv, b, x);
  };

  Events ev, tev;
  PFK_CUDA(ctx, ev.make(2, cudaEventDisableTiming));
  PFK_CUDA(ctx, tev.make(2, cudaEventDefault));

  PFK_CUDA(ctx, cudaEventRecord(tev.v[0], st));

  double bnorm = NAN, goal = NAN;
  int restarts = 0, breakdowns = 0, replacements = 0;
  SolveCtl cur = h;             // the control block as last read
  int it_known = 0;             // its iterations
  const int short_iters = M->iterations_per_step() > 1 || K < kShort ? 1 : kShort;
  int fills = 0;
  bool prev_breakdown = false;
  pfk_status result = PFK_OK;
  double rnorm_true = NAN;
  double target = NAN;
  double pass_ms = 0.0;
  double* scratch = M->scratch();

  auto true_residual = [&](double* out) -> cudaError_t {
    cudaError_t e = op_apply(op, x, scratch, b, nullptr, st);
    if (e != cudaSuccess) return e;
    e = dot_into(ctx, scratch, scratch, N, d_out, st);
    if (e != cudaSuccess) return e;
    kernel_launches += 2;
    e = cudaMemcpyAsync(h_bb + 1, d_out, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(st);
    *out = std::sqrt(h_bb[1]);
    return e;
  };
  // With profiling, one graph is in flight: after it completes, the event pairs
  // of the passes that did work (the first `done` of the K) are summed.
  auto collect = [&](int done) -> cudaError_t {
    for (int g = 0; g < done && g < K; ++g) {
      float ms = 0.f;
      cudaError_t e = cudaEventElapsedTime(&ms, pev.v[2 * g], pev.v[2 * g + 1]);
      if (e != cudaSuccess) return e;
      pass_ms += ms;
    }
    return cudaSuccess;
  };

  for (;;) {
    // ---- (re)start: pipeline fill ----
    PFK_CUDA(ctx, fill(env));
    int status = kRun;
    // iterations launched after this fill, counted from the last known total
    // (a GMRES fill forms a column, which counts too)
    int64_t reach = it_known;
    if (!profile && it_known < prm->maxit) {
      auto launch = [&](int slot) -> cudaError_t {
        // a batch: the long graph, or short ones up to K iterations or maxit
        const bool whole = giter.x && prm->maxit - reach >= (int64_t)K * M->iterations_per_step();
        const Graph& g = whole ? giter : gshort;
        const int step = whole ? K : short_iters;
        cudaError_t e = cudaSuccess;
        for (int q = 0; q < K && e == cudaSuccess && (q == 0 || reach < prm->maxit); q += step) {
          e = cudaGraphLaunch(g.x, st);
          kernel_launches += g.kernels;
          reach += (int64_t)step * M->iterations_per_step();
        }
        if (e != cudaSuccess) return e;
        e = cudaMemcpyAsync(&hc[slot], ctl, sizeof(SolveCtl), cudaMemcpyDeviceToHost, st);
        return e != cudaSuccess ? e : cudaEventRecord(ev.v[slot], st);
      };
      int q = 0;
      const bool first = !gshort.x;
      if (first) PFK_CUDA(ctx, record(gshort, short_iters, true));
      PFK_CUDA(ctx, launch(q));
      if (first) {   // while the GPU works: the fill's kernel count, and the long graph if more is to come
        PFK_CUDA(ctx, capture(cenv.st, gfill, false, [&]() -> cudaError_t { return fill(cenv); }));
        if (prm->maxit - reach >= (int64_t)K * M->iterations_per_step()) PFK_CUDA(ctx, record(giter, K, true));
      }
      for (;;) {
        const bool next = reach < prm->maxit;
        if (next) PFK_CUDA(ctx, launch(q ^ 1));
        PFK_CUDA(ctx, cudaEventSynchronize(ev.v[q]));
        if (hc[q].status != kRun) break;
        if (!next) {
          reach = hc[q].it;
          if (reach >= prm->maxit) break;
          PFK_CUDA(ctx, launch(q ^ 1));
        }
        q ^= 1;
      }
      // (a batch in flight behind this one changes nothing: its kernels see the status)
      std::memcpy(&cur, &hc[q], sizeof(SolveCtl));
    } else {
      PFK_CUDA(ctx, cudaMemcpyAsync(&hc[0], ctl, sizeof(SolveCtl), cudaMemcpyDeviceToHost, st));
      PFK_CUDA(ctx, cudaStreamSynchronize(st));
      if (!gfill.g) {
        PFK_CUDA(ctx, capture(cenv.st, gfill, false, [&]() -> cudaError_t { return fill(cenv); }));
        if (profile) PFK_CUDA(ctx, record(giter, K, true));
      }
      std::memcpy(&cur, &hc[0], sizeof(SolveCtl));
      status = cur.status;
      if (status == kRun && cur.it >= prm->maxit) {
        status = kMaxit;
      } else if (status == kRun) {
        int before = cur.passes;
        for (;;) {
          PFK_CUDA(ctx, cudaGraphLaunch(giter.x, st));
          kernel_launches += giter.kernels;
          PFK_CUDA(ctx, cudaMemcpyAsync(&hc[1], ctl, sizeof(SolveCtl), cudaMemcpyDeviceToHost, st));
          PFK_CUDA(ctx, cudaStreamSynchronize(st));
          PFK_CUDA(ctx, collect(hc[1].passes - before));
          before = hc[1].passes;
          if (hc[1].status != kRun) break;
        }
        std::memcpy(&cur, &hc[1], sizeof(SolveCtl));
        status = kRun;
      }
    }
    fills += 1;
    it_known = cur.it;
    if (std::isnan(bnorm)) {
      bnorm = std::sqrt(*h_bb);
      goal = std::fmax(prm->rtol * bnorm, prm->atol);
      target = cur.target;
    }
    if (status == kRun) status = cur.status;
    if (status == kRun && cur.it >= prm->maxit) status = kMaxit;   // a fill stopped short of its first iteration
    // (the NaN of a preconditioner application whose wait ran out reads as kNonFinite)
    if (pc && *(volatile unsigned int*)env.pcc.gave_up) status = kTimeout;
    // GMRES types: least-squares solve over the cycle's valid columns and
    // x = x_0 + U y, whatever ended the cycle
    if (gmres && status != kNonFinite && status != kTimeout) {
      PFK_CUDA(ctx, M->end_cycle(env, x));
      kernel_launches += 2;
    }
    if (status == kCycleEnd) {
      prev_breakdown = false;
      continue;
    }

    if (status == kConverged) {
      double rt = 0.0;
      PFK_CUDA(ctx, true_residual(&rt));
      rnorm_true = rt;
      if (!prm->true_residual_check || rt <= goal) {
        result = PFK_OK;
        break;
      }
      if (restarts >= prm->max_restarts) {
        set_error(ctx, "true residual above the goal after max_restarts residual replacements");
        result = PFK_ERR_NOT_CONVERGED;
        break;
      }
      replacements += 1;
      restarts += 1;
      target *= 0.5 * goal / rt;
      PFK_CUDA(ctx, cudaMemcpyAsync(&ctl->target, &target, sizeof(double), cudaMemcpyHostToDevice, st));
      prev_breakdown = false;
      continue;
    }
    if (status == kBreakdown) {
      breakdowns += 1;
      const int i_since = cur.i;
      if ((i_since <= 1 && prev_breakdown) || restarts >= prm->max_restarts) {
        set_error(ctx, "norm breakdown persisted after restarting");
        result = PFK_ERR_BREAKDOWN;
        break;
      }
      restarts += 1;
      prev_breakdown = true;
      continue;
    }
    if (status == kFillBreakdown) {
      set_error(ctx, "norm breakdown in the pipeline fill (eta_0 <= 0)");
      result = PFK_ERR_BREAKDOWN;
      break;
    }
    if (status == kNonFinite) {
      set_error(ctx, "non-finite residual norm");
      result = PFK_ERR_BREAKDOWN;
      break;
    }
    if (status == kTimeout) {   // (the inner PCG's: pc_barrier_recover replaces the message)
      set_error(ctx, "a grid-barrier wait of the persistent kernel timed out");
      result = PFK_ERR_TIMEOUT;
      break;
    }
    if (status == kMaxit) {
      set_error(ctx, "maximum number of iterations reached");
      result = PFK_ERR_NOT_CONVERGED;
      break;
    }
    set_error(ctx, "unexpected device status");
    result = PFK_ERR_CUDA;
    break;
  }
  kernel_launches += (long long)fills * gfill.kernels;
  PFK_CUDA(ctx, cudaEventRecord(tev.v[1], st));
  if (result != PFK_OK || std::isnan(rnorm_true)) {
    double rt = 0.0;
    PFK_CUDA(ctx, true_residual(&rt));
    rnorm_true = rt;
  }
  PFK_CUDA(ctx, cudaStreamSynchronize(st));
  if (pc && pc_barrier_recover(ctx, pc, st)) result = PFK_ERR_TIMEOUT;
  float ms = 0.f;
  PFK_CUDA(ctx, cudaEventElapsedTime(&ms, tev.v[0], tev.v[1]));
  const int hl = cur.hist_len;
  if (prm->history && hist_cap > 0) {
    const int ncopy = hl < hist_cap ? hl : hist_cap;
    if (ncopy > 0)
      PFK_CUDA(ctx, cudaMemcpy(prm->history, hist, (size_t)ncopy * PFK_HISTORY_FIELDS * sizeof(double),
                               cudaMemcpyDeviceToHost));
  }
  if (info) {
    info->status = result;
    info->iterations = cur.it;
    info->restarts = restarts;
    info->breakdowns = breakdowns;
    info->replacements = replacements;
    info->history_len = hl;
    info->rho0 = cur.rho0;
    info->rho_final = cur.rho;
    info->rnorm_true = rnorm_true;
    info->bnorm = bnorm;
    info->time_ms = ms;
    info->pass_launches = cur.passes;
    info->kernel_launches = (int32_t)(kernel_launches > INT32_MAX ? INT32_MAX : kernel_launches);
    info->pass_bytes = cur.alg_bytes;
    info->pass_flops = cur.alg_flops;
    info->pass_ms = profile ? pass_ms : 0.0;
  }
  return result;
}

}  // namespace pfk
