"""Failure detection of the inner PCG's single launch without a GPU fault: with no
barrier wait allowed (barrier_timeout_us < 0) the first block that has to wait
gives up, every block leaves, and the call says so; the preconditioner and the
context then work as before."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(lib):
    from paper_1511_07226_gb300 import pfk
    return pfk.Context(0)


@pytest.mark.parametrize("method", ["fcg", "gcr", "fgmres"])
@pytest.mark.parametrize("dims", [(40, 30, 20), (64, 64, 64)])
def test_inner_pcg_timeout_reported_and_usable(ctx, method, dims):
    from paper_1511_07226_gb300 import pfk
    g = W.rng(202, 1)
    n = dims[0] * dims[1] * dims[2]
    eta, b, v = 10.0 ** g.uniform(-1.0, 1.0, size=n), g.standard_normal(n), g.standard_normal(n)
    op = pfk.Operator.stencil(ctx, dims, eta)
    pc = pfk.Preconditioner(ctx, op, "inner_pcg", inner_iters=4)
    kw = dict(method=method, mmax=12, rtol=1e-9, maxit=40)
    x0, i0, _ = pfk.solve(ctx, op, pc, b, **kw)
    y0 = pc.apply(v).cpu().numpy()
    for _ in range(2):
        with pytest.raises(pfk.PfkError, match="timed out") as err:
            pfk.solve(ctx, op, pc, b, barrier_timeout_us=-1, **kw)
        assert err.value.status == -6   # PFK_ERR_TIMEOUT
        assert np.array_equal(pc.apply(v).cpu().numpy(), y0)
    x1, i1, _ = pfk.solve(ctx, op, pc, b, **kw)
    assert i1["iterations"] == i0["iterations"] and np.array_equal(x1, x0)


def test_one_block_never_waits(ctx):
    """A grid of one block has no wait that could run out."""
    from paper_1511_07226_gb300 import pfk
    op = pfk.Operator.stencil(ctx, (6, 5, 4), np.ones(120))
    pc = pfk.Preconditioner(ctx, op, "inner_pcg", inner_iters=4)
    x, info, _ = pfk.solve(ctx, op, pc, np.ones(120), method="fcg", rtol=1e-9, barrier_timeout_us=-1)
    assert info["status_name"] == "ok"
