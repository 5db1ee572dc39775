// FP64 stencil rows, one cell per thread, cells in memory order.
//
// The FP64 pipe bounds every FP64 stencil on GB300 (7 to 10 instructions per
// cell at ~76 cycles per warp instruction), and an instruction costs the same
// with one active lane as with 32.  The tiled walk (stencil.cuh) gives a warp 32
// consecutive x cells of one row, so its last tile of a row is mostly idle (nx =
// 101: 128 slots; nx = 33: 64), and its planes are separated by block barriers.
// Here a warp takes 32 consecutive cells of the whole grid, so no lane idles
// whatever the sides, and there is no barrier: the neighbours come through L1
// and L2 (11 values of 8 bytes per cell cross L2, 5.8 TB/s at the FP64 rate).
// The terms are added in the walk's order: the same result bit for bit.  Operator
// application, walk -> flat rows: 256^3 269 -> 233 us (FP64 instruction floor 222),
// 200 x 199 x 198 156 -> 119, 101 x 97 x 93 41 -> 31, 2048 x 1500 83 -> 47, 64^3
// 26 -> 22; 256^3 with advection 365 either way (floor 317).  Never slower, so
// every FP64 stencil without a sum in a pinned order takes them.
#pragma once

#include "pfk_internal.cuh"

#include <type_traits>

namespace pfk {

// I: the type of a cell index, unsigned below 2^31 cells (a row and a plane by
// multiply and shift), else unsigned long long (by division).
template <typename I>
struct FlatStencilT {
  const double* d;
  const double* kx;
  const double* ky;
  const double* kz;
  unsigned nx, ny, nz;
  I n;
  unsigned mx, my;      // c / nx = (c mx) >> sx for c < 2^31
  int sx, sy;
  double a0, a1, a2;    // upwind weights h |v_d|
  int up0, up1, up2;    // side of the upwind neighbour: -1 (v_d > 0) or +1
};

template <typename I>
inline FlatStencilT<I> flat_stencil(const pfk_operator* op) {
  FlatStencilT<I> A;
  A.d = op->d; A.kx = op->kx; A.ky = op->ky; A.kz = op->kz;
  A.nx = (unsigned)op->nx; A.ny = (unsigned)op->ny; A.nz = (unsigned)op->nz; A.n = (I)op->n;
  auto magic = [](unsigned dv, unsigned& m, int& s) {   // m = ceil(2^(31 + l) / dv), l = ceil(log2 dv): exact below 2^31
    int l = 0;
    while ((1ull << l) < dv) ++l;
    s = 31 + l;
    m = (unsigned)(((1ull << s) + dv - 1) / dv);
  };
  magic(A.nx, A.mx, A.sx);
  magic(A.ny, A.my, A.sy);
  A.a0 = op->adv[0]; A.a1 = op->adv[1]; A.a2 = op->adv[2];
  A.up0 = op->upw[0] < 0 ? -1 : 1;
  A.up1 = op->upw[1] < 0 ? -1 : 1;
  A.up2 = op->upw[2] < 0 ? -1 : 1;
  return A;
}

// Host: f(stencil, bool_constant<advection>) with the index type and the
// advection form of the operator.
template <typename F>
inline void with_flat_stencil(const pfk_operator* op, F&& f) {
  const bool adv = op->adv[0] != 0.0 || op->adv[1] != 0.0 || op->adv[2] != 0.0;
  auto go = [&](const auto& A) {
    if (adv) f(A, std::true_type{});
    else f(A, std::false_type{});
  };
  if (op->n < (int64_t)1 << 31) go(flat_stencil<unsigned>(op));
  else go(flat_stencil<unsigned long long>(op));
}

// The cells of a grid-stride loop.
#define FLAT_CELLS(I, c, n) \
  for (I c = blockIdx.x * (I)kThreads + threadIdx.x; c < (n); c += gridDim.x * (I)kThreads)

// (A m)_c; mc = m[c].
template <bool ADV, typename I>
__device__ __forceinline__ double flat_row(const FlatStencilT<I>& A, const double* __restrict__ m, I c, double& mc) {
  I row, k;
  if constexpr (sizeof(I) == 4) {
    row = (unsigned)(((unsigned long long)c * A.mx) >> A.sx);
    k = (unsigned)(((unsigned long long)row * A.my) >> A.sy);
  } else {
    row = c / A.nx;
    k = row / A.ny;
  }
  const unsigned i = (unsigned)(c - row * A.nx), j = (unsigned)(row - k * A.ny);
  const I sxy = (I)A.nx * A.ny;
  const bool xm = i > 0, xp = i + 1 < A.nx, ym = j > 0, yp = j + 1 < A.ny;
  mc = m[c];
  const double d = A.d[c], kx = A.kx[c], ky = A.ky[c];
  const double mxm = xm ? m[c - 1] : 0.0, kxm = xm ? A.kx[c - 1] : 0.0, mxp = xp ? m[c + 1] : 0.0;
  const double mym = ym ? m[c - A.nx] : 0.0, kym = ym ? A.ky[c - A.nx] : 0.0, myp = yp ? m[c + A.nx] : 0.0;
  double mzm = 0.0, kzm = 0.0, mzp = 0.0, kz = 0.0;
  if (A.nz > 1) {
    kz = A.kz[c];
    if (k > 0) {
      mzm = m[c - sxy];
      kzm = A.kz[c - sxy];
    }
    if (k + 1 < A.nz) mzp = m[c + sxy];
  }
  double y = d * mc;
  y -= kxm * mxm;
  y -= kx * mxp;
  y -= kym * mym;
  y -= ky * myp;
  if (A.nz > 1) {
    y -= kzm * mzm;
    y -= kz * mzp;
  }
  if (ADV) {
    y -= A.a0 * (A.up0 < 0 ? mxm : mxp);
    y -= A.a1 * (A.up1 < 0 ? mym : myp);
    if (A.nz > 1) y -= A.a2 * (A.up2 < 0 ? mzm : mzp);
  }
  return y;
}

}  // namespace pfk
