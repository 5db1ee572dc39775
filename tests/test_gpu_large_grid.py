"""An operator of more than 2^31 cells, whose cells are indexed in 64 bits (about
130 GB on the device).  Integer values and unit viscosity: every row is exact."""
import pytest

pytestmark = pytest.mark.gpu


def test_apply_beyond_2_31_cells(lib):
    import torch
    from paper_1511_07226_gb300 import pfk
    N = 1300
    n = N ** 3
    assert n > 1 << 31
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 170 * (1 << 30):
        pytest.skip("needs 170 GiB of free device memory")
    ctx = pfk.Context(0)
    eta = torch.ones(n, device="cuda", dtype=torch.float64)
    op = pfk.Operator.stencil(ctx, (N, N, N), eta)
    del eta
    torch.cuda.empty_cache()
    x = (torch.arange(n, device="cuda", dtype=torch.int64).remainder_(7)).double()
    y = op.apply(x).reshape(N, N, N)
    x = x.reshape(N, N, N)
    for k in (1, N // 2, 1271, N - 2):   # 1271: planes on both sides of cell 2^31
        ref = 6 * x[k, 1:-1, 1:-1] - x[k - 1, 1:-1, 1:-1] - x[k + 1, 1:-1, 1:-1] - x[k, :-2, 1:-1] - x[k, 2:, 1:-1] \
            - x[k, 1:-1, :-2] - x[k, 1:-1, 2:]
        assert torch.equal(y[k, 1:-1, 1:-1], ref)
    # a corner has three half-distance Dirichlet faces: diagonal 3 * 2 + 3
    assert float(y[-1, -1, -1]) == 9 * float(x[-1, -1, -1]) - float(x[-2, -1, -1] + x[-1, -2, -1] + x[-1, -1, -2])
    del x, y, op, ctx
    torch.cuda.empty_cache()
