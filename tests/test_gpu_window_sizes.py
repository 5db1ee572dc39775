"""The window dots of FCG, GCR and FGMRES with windows that really fill: mmax + 3
iterations (FGMRES: one cycle of mmax), for mmax at both ends of every size the
loop is instantiated for above 16 slots (20, 24, 28, 32), against the oracle.
(PIPEGCR's, with windows up to 32, are among the recorded results.)

Tolerance: an iteration rounds each of its ~10 vector and window operations to
2^-53 of their terms; the blocking methods form residuals and directions anew, so
35 iterations at a diagonally scaled condition of about 1e3 move the iterate by
less than 35 x 10 x 1.1e-16 x 1e3 < 1e-10."""
import numpy as np
import pytest

import workloads as W
from oracle import krylov as K
from oracle import operators as O
from oracle import preconditioners as PC

pytestmark = pytest.mark.gpu

DIMS = (17, 15, 13)


@pytest.fixture(scope="module")
def ctx(lib):
    from paper_1511_07226_gb300 import pfk
    return pfk.Context(0)


@pytest.mark.parametrize("method", ["gcr", "fgmres", "fcg"])
@pytest.mark.parametrize("mmax", [17, 20, 21, 24, 25, 28, 29, 32])
def test_full_windows(ctx, method, mmax):
    from paper_1511_07226_gb300 import pfk
    g = W.rng(203, 1)
    n = DIMS[0] * DIMS[1] * DIMS[2]
    eta, b = 10.0 ** g.uniform(-1.0, 1.0, size=n), g.standard_normal(n)
    aop = O.StencilOperator(DIMS, eta)
    op = pfk.Operator.stencil(ctx, DIMS, eta)
    pc = pfk.Preconditioner(ctx, op, "jacobi")
    its = mmax if method == "fgmres" else mmax + 3
    ref = K.solve(method, aop.apply, PC.JacobiPC(aop), b, prm=K.Params(mmax=mmax, rtol=1e-14, maxit=its))
    x, info, _ = pfk.solve(ctx, op, pc, b, method=method, mmax=mmax, rtol=1e-14, maxit=its)
    assert info["iterations"] == ref.iterations == its     # the last windows held mmax vectors
    assert np.linalg.norm(x - ref.x) <= 1e-10 * np.linalg.norm(ref.x)
