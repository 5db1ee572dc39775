// FP64 inner Jacobi-PCG (Alg. 3, M^-1 = D^-1) in one cooperative launch, for
// grids whose inner vectors fit in the SMs' shared memory.
//
// As separate kernels (pc.cu) an application of k inner iterations is 3k
// launches.  Below about a million cells each of them spends most of its time
// outside its loop: launch and block ramp-up, the L2 round trips of its control
// words, the sums and the last-block combine (64^3: 12 kernels of 4 to 15 us for
// 27 us of FP64 work).  Here every SM keeps one block with a
// fixed range of consecutive cells; r, s (D^-1 r after the r update), x and p of
// those cells stay in shared memory for the whole application, p also in global
// memory for the stencils of the neighbouring blocks, and the blocks meet at a
// grid barrier where the algorithm needs a grid-wide result: three per inner
// iteration (<s, p>, <D^-1 r, r>, p complete).  A reduction writes one partial
// sum per block before its barrier; after it every block adds all partial sums
// in the same order, so all hold bitwise the same scalars.  The statements per
// cell are those of the separate kernels; the sums are added in another order,
// so single applications and the blocking methods (FCG, GCR, FGMRES) use this
// form and the pipelined methods, which amplify that difference, do not
// (PcCall::pinned).
//
// A barrier and the sum behind it take 3 to 4 us, in which the warps that do
// not wait have nothing to do, so work that depends on neither is placed there:
// the x update during the sum for gamma, and the x and y terms of the stencil
// while p becomes complete everywhere (64^3, four inner iterations: 90.5 ->
// 88 -> 85 us; 101 x 97 x 93: 146 -> 140 us).  The registers are kept to two
// blocks per SM although a launch has one, so that the applications of two
// solves on different streams run side by side: with all registers for one
// block 64^3 takes 83 us, but a burst of eight small solves on four workers, all
// with this form, 29 ms instead of 21.
//
// Every wait is bounded (pfk_solve_params' barrier_timeout_us, else 2 s): a wait
// that runs out raises an abort word that ends all other waits, the blocks that
// saw it write NaN, and a host-pinned word tells the host, which reports
// PFK_ERR_TIMEOUT and resets the barrier words before the next application.
#include "pfk_internal.cuh"

#include <cstddef>

namespace pfk {

constexpr int kResThreads = 512;
constexpr int kResSmemLimit = 220 * 1024;         // dynamic shared memory of a block (of 227 KB in all)
constexpr int kResCellBytes = 4 * 8 + 1;          // r, s, x, p and the neighbour flags
constexpr int kResMinCells = 256;                 // cells per block before the grid is grown

struct ResArgs {
  const double* d;
  const double* kx;
  const double* ky;
  const double* kz;
  const double* dinv;
  int nx, ny, nz;
  double a0, a1, a2;
  int u0, u1, u2;
  int64_t n;
  const double* v;
  const double* add;
  double* out;
  double* p;            // global copy of p
  double* partials;     // 2 gridDim
  PcCtl* ctl;
  int k;
  const int* status;
  long long bar_timeout_ns;
  unsigned int* gave_up;   // host-pinned
};

namespace {

__device__ __forceinline__ unsigned res_ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long res_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Thread 0's part of the grid barrier (the block's writes are ordered before it
// by a block barrier): arrive with acquire-release; the last arrival resets the
// counter and releases the next generation.  `gen` is the generation before
// this barrier, counted by the caller, so arriving needs no load, and a wait
// polls one word: reading the timer and the abort word on every poll as well
// tripled the time to notice a release.  False when a wait gave up.
__device__ __forceinline__ bool res_arrive_wait(const ResArgs& a, unsigned gen) {
  PcCtl* ctl = a.ctl;
  unsigned old;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(&ctl->bar_count) : "memory");
  if (old == gridDim.x - 1) {
    ctl->bar_count = 0u;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->bar_gen) : "memory");
    return true;
  }
  unsigned long long t0 = 0ull;
  for (unsigned polls = 1; res_ld_acquire(&ctl->bar_gen) == gen; ++polls) {
    if ((polls & 63u) && a.bar_timeout_ns > 0) continue;
    if (res_ld_acquire(&ctl->bar_abort)) return false;
    const unsigned long long t = res_ns();
    if (t0 == 0ull) t0 = t;
    if (a.bar_timeout_ns <= 0 || t - t0 > (unsigned long long)a.bar_timeout_ns) {
      atomicExch(&ctl->bar_abort, 1u);
      return false;
    }
  }
  return true;
}

struct ResShared {
  double buf[kResThreads];
  double part[4];
  double sum, quot;
  unsigned gen;        // barriers passed (thread 0)
  int ok;
};

// Grid barrier; false when a wait gave up (all threads of the block agree).
// meanwhile(t, nt), t < nt, runs in the other warps while warp 0 waits.
template <typename G>
__device__ __forceinline__ bool res_barrier(const ResArgs& a, ResShared& sh, G&& meanwhile) {
  __syncthreads();
  if (threadIdx.x >= 32) meanwhile((int)threadIdx.x - 32, kResThreads - 32);
  else if (threadIdx.x == 0) sh.ok = res_arrive_wait(a, sh.gen++);
  __syncthreads();
  return sh.ok != 0;
}

// Grid-wide sum of `acc` into sh.sum, with the barrier's guarantees, and sh.quot
// = quot(sum).  Block: the first four warps (one per SM sub-partition) add the
// sixteen warps' values lane by lane and run one shuffle tree each.  Grid: lane
// l of warp 0 takes the blocks l, l + 32, ..., then a shuffle tree.  One thread
// forms the quotient (a division is a chain of FP64 instructions; in all sixteen
// warps it held the FP64 pipes for 1.5 us).  parity alternates from one sum to
// the next, so a block that runs ahead never overwrites a partial sum that
// another still reads.  meanwhile(t, nt), t < nt, runs in the warps of
// the three sub-partitions that warp 0 is not on, while it waits and combines.
template <typename F, typename G>
__device__ __forceinline__ bool res_sum(const ResArgs& a, ResShared& sh, double acc, int parity, F&& quot,
                                        G&& meanwhile) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  sh.buf[threadIdx.x] = acc;
  __syncthreads();
  if (warp < 4) {
    const double* b = sh.buf + warp * 128 + lane;
    const double s = warp_sum((b[0] + b[32]) + (b[64] + b[96]));
    if (lane == 0) sh.part[warp] = s;
  }
  __syncthreads();
  double* part = a.partials + (size_t)parity * gridDim.x;
  if (warp == 0) {
    int ok = 1;
    if (lane == 0) {
      part[blockIdx.x] = (sh.part[0] + sh.part[1]) + (sh.part[2] + sh.part[3]);
      ok = res_arrive_wait(a, sh.gen++);
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    double t[8];
    double s = 0.0;
    for (int b0 = 0; b0 < (int)gridDim.x; b0 += 256) {
#pragma unroll
      for (int u = 0; u < 8; ++u) t[u] = b0 + 32 * u + lane < (int)gridDim.x ? __ldcg(&part[b0 + 32 * u + lane]) : 0.0;
      s += ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
    }
    s = warp_sum(s);
    if (lane == 0) {
      sh.sum = s;
      sh.quot = quot(s);
      sh.ok = ok;
    }
  } else if (warp & 3) {
    meanwhile(((warp >> 2) * 3 + (warp & 3) - 1) * 32 + lane, kResThreads / 4 * 3);
  }
  __syncthreads();
  return sh.ok != 0;
}

}  // namespace

template <bool ADV>
__global__ void __launch_bounds__(kResThreads, 2) pcg_resident_kernel(ResArgs a) {
  if (a.status && *a.status != kRun) return;
  extern __shared__ double res_smem[];
  __shared__ ResShared sh;
  const int64_t lo64 = a.n * blockIdx.x / gridDim.x, hi64 = a.n * (blockIdx.x + 1) / gridDim.x;
  const int cells = (int)(hi64 - lo64), lo = (int)lo64;
  const int cap = (int)((a.n + gridDim.x - 1) / gridDim.x);
  double* r = res_smem;
  double* s = r + cap;
  double* x = s + cap;
  double* p = x + cap;
  unsigned char* nb = reinterpret_cast<unsigned char*>(p + cap);   // which neighbours exist: -x, +x, -y, +y, -z, +z
  const int nx = a.nx, sxy = a.nx * a.ny;
  if (threadIdx.x == 0) {
    sh.gen = res_ld_acquire(&a.ctl->bar_gen);   // no block passes the first barrier before this one arrives
    sh.part[0] = res_ld_acquire(&a.ctl->bar_abort) ? 1.0 : 0.0;
  }
  __syncthreads();
  // an earlier application gave up: the barrier words are not usable
  bool ok = sh.part[0] == 0.0;
  __syncthreads();

  // Terms of (A p)_q up to the y neighbours, in the walk's order.  They are
  // formed before the barrier that completes p, while it is waited for, for the
  // cells whose x and y neighbours lie in the block (all but its first and last
  // nx cells), and kept in s; the z and advection terms follow after it.
  auto at = [&](int q, int o) { return (unsigned)(q + o) < (unsigned)cells ? p[q + o] : __ldcg(&a.p[lo + q + o]); };
  auto xy_terms = [&](int q) {
    const int c = lo + q;
    const unsigned f = nb[q];
    const double mxm = (f & 1u) ? at(q, -1) : 0.0, kxm = (f & 1u) ? a.kx[c - 1] : 0.0;
    const double mxp = (f & 2u) ? at(q, 1) : 0.0;
    const double mym = (f & 4u) ? at(q, -nx) : 0.0, kym = (f & 4u) ? a.ky[c - nx] : 0.0;
    const double myp = (f & 8u) ? at(q, nx) : 0.0;
    double y = a.d[c] * p[q];
    y -= kxm * mxm;
    y -= a.kx[c] * mxp;
    y -= kym * mym;
    y -= a.ky[c] * myp;
    return y;
  };
  auto inner_terms = [&](int t, int nt) {
#pragma unroll 2
    for (int q = nx + t; q < cells - nx; q += nt) s[q] = xy_terms(q);
  };

  // r_0 = v, p_0 = D^-1 r_0, gamma_0 = <D^-1 r_0, r_0>
  double acc = 0.0;
  for (int q = threadIdx.x; q < cells; q += kResThreads) {
    const int c = lo + q, i = c % nx, row = c / nx, j = row % a.ny, kk = row / a.ny;
    nb[q] = (unsigned char)((i > 0 ? 1 : 0) | (i < nx - 1 ? 2 : 0) | (j > 0 ? 4 : 0) | (j < a.ny - 1 ? 8 : 0) |
                            (kk > 0 ? 16 : 0) | (kk < a.nz - 1 ? 32 : 0));
    const double rv = a.v[c], z = a.dinv[c] * rv;
    r[q] = rv;
    p[q] = z;
    x[q] = 0.0;
    a.p[c] = z;
    acc = fma(z, rv, acc);
  }
  ok = ok && res_sum(a, sh, acc, 0, [](double) { return 0.0; }, inner_terms);
  double gamma = sh.sum, alpha = 0.0;
  int parity = 1;
  bool last = false;     // the final x still needs alpha p
  if (ok && gamma != 0.0) {
    for (int it = 0; it < a.k; ++it) {
      // s_i = A p_i (the walk's order of terms), eta_i = <s_i, p_i>
      acc = 0.0;
#pragma unroll 2
      for (int q = threadIdx.x; q < cells; q += kResThreads) {
        const int c = lo + q;
        const unsigned f = nb[q];
        const double mc = p[q];
        double mzm = 0.0, kzm = 0.0, mzp = 0.0, kzc = 0.0;
        if (a.nz > 1) {
          kzc = a.kz[c];
          if (f & 16u) { mzm = at(q, -sxy); kzm = a.kz[c - sxy]; }
          if (f & 32u) mzp = at(q, sxy);
        }
        double y = q >= nx && q < cells - nx ? s[q] : xy_terms(q);
        if (a.nz > 1) {
          y -= kzm * mzm;
          y -= kzc * mzp;
        }
        if (ADV) {
          y -= a.a0 * ((f & (a.u0 < 0 ? 1u : 2u)) ? at(q, a.u0 < 0 ? -1 : 1) : 0.0);
          y -= a.a1 * ((f & (a.u1 < 0 ? 4u : 8u)) ? at(q, a.u1 < 0 ? -nx : nx) : 0.0);
          if (a.nz > 1) y -= a.a2 * (a.u2 < 0 ? mzm : mzp);
        }
        s[q] = y;
        acc = fma(y, mc, acc);
      }
      if (!(ok = res_sum(a, sh, acc, parity, [=](double eta) { return gamma / eta; }, [](int, int) {}))) break;
      parity ^= 1;
      if (sh.sum == 0.0) break;      // eta_i
      alpha = sh.quot;
      if (it + 1 == a.k) {
        last = true;
        break;
      }
      // x_{i+1}, r_{i+1}, z = D^-1 r_{i+1} (kept in s), gamma_{i+1} = <z, r_{i+1}>
      acc = 0.0;
#pragma unroll 4
      for (int q = threadIdx.x; q < cells; q += kResThreads) {
        const double rv = fma(-alpha, s[q], r[q]), z = a.dinv[lo + q] * rv;
        r[q] = rv;
        s[q] = z;
        acc = fma(z, rv, acc);
      }
      // nothing waits for x: its update fills the FP64 pipes during the reduction
      ok = res_sum(a, sh, acc, parity, [=](double g) { return g / gamma; }, [&](int t, int nt) {
#pragma unroll 4
        for (int q = t; q < cells; q += nt) x[q] = fma(alpha, p[q], x[q]);
      });
      if (!ok) break;
      parity ^= 1;
      if (sh.sum == 0.0) break;      // gamma_{i+1}
      const double beta = sh.quot;
      gamma = sh.sum;
#pragma unroll 4
      for (int q = threadIdx.x; q < cells; q += kResThreads) {
        const double pv = fma(beta, p[q], s[q]);
        p[q] = pv;
        a.p[lo + q] = pv;
      }
      if (!(ok = res_barrier(a, sh, inner_terms))) break;
    }
  }
  if (!ok && threadIdx.x == 0) {
    *(volatile unsigned int*)a.gave_up = 1u;
    __threadfence_system();
  }
  // out = add + x_k
#pragma unroll 4
  for (int q = threadIdx.x; q < cells; q += kResThreads) {
    double y = x[q];
    if (last) y = fma(alpha, p[q], y);
    if (!ok) y = nan("");
    a.out[lo + q] = a.add ? a.add[lo + q] + y : y;
  }
}

static int res_blocks(const pfk_context* ctx, int64_t n) {
  const int64_t need = (n + kResMinCells - 1) / kResMinCells;
  return (int)(need < ctx->num_sms ? need : ctx->num_sms);
}

static size_t res_smem_bytes(const pfk_context* ctx, int64_t n) {
  const int64_t g = res_blocks(ctx, n), cap = (n + g - 1) / g;
  return (size_t)(cap * kResCellBytes + 8);
}

// Whether the resident form applies: the cells of a block fit in its shared
// memory (152 SMs: up to about 1.03 M cells) and the partial sums in the
// preconditioner's.  It is the faster form at every size it can hold (four inner
// iterations, separate kernels -> one launch: 24^3 100 -> 61 us, 64^3 133 -> 92,
// 96^3 192 -> 147, before the work in the waits), so the memory sets the line.
bool pcg_resident_fits(const pfk_pc* pc) {
  const int64_t n = pc->op->n;
  return n >= 1 && n < INT32_MAX / 2 && res_smem_bytes(pc->ctx, n) <= (size_t)kResSmemLimit &&
         2 * res_blocks(pc->ctx, n) <= pc->partials_cap;
}

cudaError_t pcg_resident(const pfk_pc* pc, const double* v, double* out, const double* add, const int* status,
                         cudaStream_t st, const PcCall& how) {
  const pfk_operator* op = pc->op;
  ResArgs a;
  a.d = op->d; a.kx = op->kx; a.ky = op->ky; a.kz = op->kz; a.dinv = op->dinv;
  a.nx = op->nx; a.ny = op->ny; a.nz = op->nz;
  a.a0 = op->adv[0]; a.a1 = op->adv[1]; a.a2 = op->adv[2];
  a.u0 = op->upw[0]; a.u1 = op->upw[1]; a.u2 = op->upw[2];
  a.n = op->n;
  a.v = v; a.add = add; a.out = out;
  a.p = (double*)pc->buf;
  a.partials = pc->partials;
  a.ctl = pc->ctl;
  a.k = pc->inner;
  a.status = status;
  a.bar_timeout_ns = how.bar_timeout_ns;
  a.gave_up = how.gave_up;
  const bool adv = op->adv[0] != 0.0 || op->adv[1] != 0.0 || op->adv[2] != 0.0;
  const void* fn = adv ? (const void*)pcg_resident_kernel<true> : (const void*)pcg_resident_kernel<false>;
  const int smem = (int)res_smem_bytes(pc->ctx, a.n);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmemLimit);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(res_blocks(pc->ctx, a.n));
  cfg.blockDim = dim3(kResThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* params[] = {&a};
  return cudaLaunchKernelExC(&cfg, fn, params);
}

bool pc_barrier_recover(pfk_context* ctx, const pfk_pc* pc, cudaStream_t st) {
  volatile unsigned int* w = &ctx->pinned->pc_gave_up;
  if (!*w) return false;
  *w = 0u;
  static_assert(offsetof(PcCtl, bar_pad) == offsetof(PcCtl, bar_count) + 3 * sizeof(unsigned int), "one range");
  if (pc->ctl) cudaMemsetAsync(&pc->ctl->bar_count, 0, 4 * sizeof(unsigned int), st);
  set_error(ctx, "a grid-barrier wait of the inner PCG timed out");
  return true;
}

}  // namespace pfk
