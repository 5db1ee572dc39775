"""The FP64 inner Jacobi-PCG in one cooperative launch and the flat FP64 stencil
rows, at the sizes where their decompositions change: one cell per block and
the last block shorter, the 256-cell minimum per block (152 SMs: 38,912 cells),
lines and planes without z or y neighbours, ragged rows, and both sides of the
largest resident size (about 1.03 M cells at 152 SMs), where the separate
kernels take over.

Tolerance: every FP64 operation of k inner iterations contributes a relative
rounding of 2^-53 = 1.1e-16; sums of n <= 1.1e6 products in any order differ by
at most ~log2(n) = 20 such roundings of their terms' magnitudes, and k = 4
iterations of a Jacobi-scaled operator (contrast 1e2) amplify them by less than
a factor 1e2: 20 x 1.1e-16 x 1e2 x 4 < 1e-12, the bound of the other inner-PCG
parity tests."""
import numpy as np
import pytest

import workloads as W
from oracle import operators as O
from oracle import preconditioners as PC

pytestmark = pytest.mark.gpu

NONE, ADV = (0.0, 0.0, 0.0), (2.0, 1.0, -1.0)


@pytest.fixture(scope="module")
def ctx(lib):
    from paper_1511_07226_gb300 import pfk
    return pfk.Context(0)


def _problem(dims, item):
    g = W.rng(201, item)
    n = dims[0] * dims[1] * dims[2]
    return 10.0 ** g.uniform(-1.0, 1.0, size=n), g.standard_normal(n)


@pytest.mark.parametrize("dims,vel,k", [
    ((1, 1, 1), NONE, 4), ((7, 1, 1), NONE, 2), ((1, 1, 300), NONE, 4), ((33, 5, 1), NONE, 1),
    ((257, 3, 1), ADV, 3), ((19, 13, 11), ADV, 4), ((64, 32, 19), NONE, 4), ((38913, 1, 1), NONE, 4),
    ((101, 97, 93), NONE, 4), ((101, 101, 101), ADV, 2), ((128, 104, 96), NONE, 2)])
def test_inner_pcg_sizes(ctx, dims, vel, k):
    from paper_1511_07226_gb300 import pfk
    eta, v = _problem(dims, 1)
    aop = O.StencilOperator(dims, eta, vel)
    op = pfk.Operator.stencil(ctx, dims, eta, vel)
    pc = pfk.Preconditioner(ctx, op, "inner_pcg", inner_iters=k)
    ref = PC.InnerPCG(aop, k)(v)
    got = pc.apply(v).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    assert np.array_equal(pc.apply(v).cpu().numpy(), got)


def test_inner_pcg_early_exit_and_nan(ctx):
    """v = 0 returns 0; a one-cell operator is solved exactly by the first inner
    iteration; a NaN input gives NaN and leaves the preconditioner usable."""
    from paper_1511_07226_gb300 import pfk
    dims = (40, 30, 20)
    eta, v = _problem(dims, 2)
    op = pfk.Operator.stencil(ctx, dims, eta)
    pc = pfk.Preconditioner(ctx, op, "inner_pcg", inner_iters=4)
    assert np.array_equal(pc.apply(np.zeros(op.n)).cpu().numpy(), np.zeros(op.n))
    v[17] = np.nan
    assert np.isnan(pc.apply(v).cpu().numpy()).all()
    v[17] = 1.0
    assert np.isfinite(pc.apply(v).cpu().numpy()).all()
    one = pfk.Operator.stencil(ctx, (1, 1, 1), np.array([3.0]))
    got = pfk.Preconditioner(ctx, one, "inner_pcg", inner_iters=5).apply(np.array([2.0])).cpu().numpy()
    assert np.allclose(got * O.StencilOperator((1, 1, 1), np.array([3.0])).diagonal(), 2.0, rtol=1e-14)


@pytest.mark.parametrize("dims,vel", [
    ((1, 1, 1), NONE), ((31, 1, 1), ADV), ((1, 33, 1), ADV), ((1, 1, 257), ADV), ((255, 3, 2), ADV),
    ((33, 33, 33), NONE), ((129, 65, 17), ADV), ((2048, 3, 1), ADV)])
def test_flat_stencil_sizes(ctx, dims, vel):
    """A x entry by entry: at most 10 roundings of the terms of a row."""
    from paper_1511_07226_gb300 import pfk
    eta, v = _problem(dims, 3)
    aop = O.StencilOperator(dims, eta, vel)
    ref = aop.apply(v)
    scale = np.abs(aop.diagonal()).max() * np.abs(v).max()
    got = pfk.Operator.stencil(ctx, dims, eta, vel).apply(v).cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 2e-14 * scale
    cheb = pfk.Preconditioner(ctx, pfk.Operator.stencil(ctx, dims, eta, vel), "chebyshev", inner_iters=3)
    cref = PC.Chebyshev(aop, 3)(v)
    assert np.linalg.norm(cheb.apply(v).cpu().numpy() - cref) <= 1e-12 * np.linalg.norm(cref)


@pytest.mark.parametrize("method", ["gcr", "pipegcr", "fgmres", "fcg"])
@pytest.mark.parametrize("mmax", [3, 4, 5, 8, 12, 13, 17, 21, 25, 32])
def test_window_dots_sizes(ctx, method, mmax):
    """Windows on both sides of every rounded size of the window-dots loop:
    iterations of a well-conditioned problem against the oracle (strict: the
    recurrences have not amplified rounding yet)."""
    from oracle import krylov as K
    from paper_1511_07226_gb300 import pfk
    dims = (17, 15, 13)
    eta, b = _problem(dims, 4)
    eta = eta ** 0.25
    aop = O.StencilOperator(dims, eta)
    op = pfk.Operator.stencil(ctx, dims, eta)
    pc = pfk.Preconditioner(ctx, op, "jacobi")
    its = min(mmax + 3, 18) if method != "fgmres" else min(mmax, 18)
    prm = K.Params(mmax=mmax, rtol=1e-14, maxit=its)
    ref = K.solve(method, aop.apply, PC.JacobiPC(aop), b, prm=prm)
    x, info, hist = pfk.solve(ctx, op, pc, b, method=method, mmax=mmax, rtol=1e-14, maxit=its, history=64)
    assert info["iterations"] == ref.iterations
    assert np.linalg.norm(x - ref.x) <= 1e-10 * np.linalg.norm(ref.x)


@pytest.mark.parametrize("exponent", [-510, -490, 490, 505])
def test_single_launch_pipefcg_extreme_scales(ctx, exponent):
    """eta_k ~ scale^2 outside the range whose reciprocals are kept (2^-1000 ..
    2^1000), against the one-kernel-per-step path at the same scale (its dots
    meet the same subnormal products): a few units of 2^-53 per iteration,
    amplified by 8 iterations at contrast 1e3 by less than 1e4:
    8 x 4 x 1.1e-16 x 1e4 < 1e-10."""
    from paper_1511_07226_gb300 import pfk
    c = W.poisson2d_inclusions()
    op = pfk.Operator.stencil(ctx, c["dims"], c["eta"], storage="csr")
    pc = pfk.Preconditioner(ctx, op, "jacobi")
    kw = dict(method="pipefcg", mmax=30, rtol=1e-14, maxit=8)
    b = np.ldexp(np.asarray(c["b"], dtype=np.float64), exponent)
    x0, i0, _ = pfk.solve(ctx, op, pc, b, persistent="off", **kw)
    x1, i1, _ = pfk.solve(ctx, op, pc, b, persistent="on", **kw)
    assert i0["iterations"] == i1["iterations"] == 8
    x0, x1 = np.ldexp(x0, -exponent), np.ldexp(x1, -exponent)
    assert np.linalg.norm(x1 - x0) <= 1e-10 * np.linalg.norm(x0)
