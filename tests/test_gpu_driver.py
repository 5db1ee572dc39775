"""Launches of the solve driver: none without iterations to do."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(lib):
    from paper_1511_07226_gb300 import pfk
    return pfk.Context(0)


@pytest.mark.parametrize("method", ["pipefcg", "fcg"])
def test_single_launch_solve_enqueues_only_working_launches(ctx, method):
    """The single-launch kernel does 16 iterations per launch, so maxit
    iterations (out of the tolerance's reach) take ceil(maxit / 16) launches
    beside those of the fill and the norms, whatever the graph length."""
    from paper_1511_07226_gb300 import pfk
    c = W.poisson2d_inclusions()
    op = pfk.Operator.stencil(ctx, c["dims"], c["eta"], storage="csr")
    pc = pfk.Preconditioner(ctx, op, "jacobi")

    def launches(maxit, **kw):
        x, info, _ = pfk.solve(ctx, op, pc, c["b"], method=method, mmax=30, rtol=1e-15, maxit=maxit,
                               persistent="on", **kw)
        assert info["iterations"] == maxit and np.isfinite(x).all()
        return info["kernel_launches"]

    one = launches(16)
    for maxit in (1, 17, 48, 49, 200, 320):
        assert launches(maxit) - one == -(-maxit // 16) - 1, maxit
    assert launches(48, graph_iters=1) == launches(48)
