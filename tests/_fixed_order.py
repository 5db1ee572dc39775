"""Solves whose results are pinned bit for bit, and the recording of them.

The pipelined recurrences (PIPEFCG, PIPEGCR, PIPEFGMRES and their variants)
never form a residual or a preconditioned residual anew, so a last-bit
difference of one inner product grows within some tens of iterations: 26^3
PIPEGCR at contrast 1e3 moves by up to 5e-7 in 20.  With a preconditioner that
rounds its input to FP32 the blocking methods' iterates move too, by up to the
FP32 rounding.  The order in which these kernels add is therefore part of
their results.  Inputs are exact (integers and
powers of two): the same bits wherever they are made.

`python tests/_fixed_order.py OUT.json` (repository root as the working folder, a
GPU, the library built) records the results that tests/test_gpu_fixed_order.py
compares with; the recorded ones were made on a GB300 (152 SMs, which the grids
and so the orders depend on) by the build of commit c2a6e66.
"""
import json
import os
import sys

import numpy as np

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fixed_order.json")
SAMPLES = 33
NONE, ADV = (0.0, 0.0, 0.0), (2.0, 1.0, -1.0)


def _c(group, method, dims, mmax, maxit, pc="inner_pcg", inner=4, vel=NONE, storage="matrix_free", **kw):
    return dict(group=group, method=method, dims=dims, mmax=mmax, maxit=maxit, pc=pc, inner=inner, vel=vel,
                storage=storage, **kw)


CASES = {
    # the FP64 inner PCG: one cell per thread, several, a grid larger than shared memory, 2D, advection, k = 1
    "pcg_24": _c("pcg", "pipefcg", (24, 20, 18), 30, 24),
    "pcg_64": _c("pcg", "pipefcg", (64, 60, 44), 30, 16),
    "pcg_101": _c("pcg", "pipefcg", (101, 97, 93), 8, 12),
    "pcg_150": _c("pcg", "pipefcg", (150, 92, 85), 16, 10),
    "pcg_2d": _c("pcg", "pipefcg", (300, 210, 1), 30, 16, inner=5),
    "pcg_line": _c("pcg", "pipefcg", (2000, 1, 1), 30, 12, inner=1),
    "pcg_naive": _c("pcg", "pipefcg_naive", (40, 33, 21), 30, 12),
    "pcg_gcr_w": _c("pcg", "pipegcr_w", (40, 33, 21), 30, 12),
    "pcg_theta": _c("pcg", "pipefcg_theta", (40, 33, 21), 30, 12),
    "pcg_adv": _c("pcg", "pipefgmres", (48, 40, 36), 14, 14, inner=3, vel=ADV),
    # PIPEGCR: windows up to 32, the three instantiations, ragged sides, 2D, advection
    "gcr_64": _c("pipegcr", "pipegcr", (64, 64, 64), 32, 34, pc="jacobi"),
    "gcr_24": _c("pipegcr", "pipegcr", (24, 20, 18), 30, 24),
    "gcr_ragged": _c("pipegcr", "pipegcr", (101, 67, 45), 16, 20, pc="jacobi"),
    "gcr_8": _c("pipegcr", "pipegcr", (33, 35, 37), 8, 12),
    "gcr_150": _c("pipegcr", "pipegcr", (150, 92, 85), 23, 24, pc="jacobi"),
    "gcr_2d": _c("pipegcr", "pipegcr", (300, 210, 1), 30, 16),
    "gcr_adv": _c("pipegcr", "pipegcr", (48, 40, 36), 30, 18, vel=ADV),
    # the grouped kernel
    "grp_fcg": _c("grouped", "pipefcg", [(26, 26, 26), (40, 37, 33), (31, 17, 5), (64, 9, 1)], 30, 16),
    "grp_gcr": _c("grouped", "pipegcr", [(26, 26, 26), (40, 37, 33), (31, 17, 5), (64, 9, 1)], 30, 16),
    "grp_gmres": _c("grouped", "pipefgmres", [(26, 26, 26), (40, 37, 33), (31, 17, 5)], 12, 12, vel=ADV),
    # the single-launch PIPEFCG on an assembled operator
    "csr_4": _c("csr", "pipefcg", (64, 64, 1), 4, 24, pc="jacobi", storage="csr"),
    "csr_8": _c("csr", "pipefcg", (125, 139, 1), 8, 20, pc="jacobi", storage="csr"),
    "csr_16": _c("csr", "pipefcg", (64, 64, 1), 16, 24, pc="jacobi", storage="csr"),
    "csr_30": _c("csr", "pipefcg", (64, 64, 1), 30, 48, pc="jacobi", storage="csr"),
    "csr_32": _c("csr", "pipefcg", (125, 139, 1), 32, 40, pc="none", storage="csr"),
    # FCG, GCR and FGMRES with a preconditioner in reduced precision
    "prec_fcg": _c("prec", "fcg", (64, 60, 44), 30, 34, precision="fp32"),
    "prec_fcg_150": _c("prec", "fcg", (150, 92, 85), 16, 18, precision="bf16"),
    "prec_fcg_8": _c("prec", "fcg", (33, 35, 37), 8, 12, pc="chebyshev", precision="bf16"),
    "prec_fcg_csr": _c("prec", "fcg", (48, 40, 36), 30, 16, precision="fp32", storage="csr"),
    "prec_gcr": _c("prec", "gcr", (64, 60, 44), 32, 34, precision="fp32"),
    "prec_gcr_adv": _c("prec", "gcr", (48, 40, 36), 12, 16, pc="chebyshev", vel=ADV, precision="bf16"),
    "prec_gcr_csr": _c("prec", "gcr", (300, 210, 1), 30, 16, precision="fp32", storage="csr"),
    "prec_fgmres": _c("prec", "fgmres", (118, 112, 127), 25, 25, pc="chebyshev", inner=8, vel=ADV, precision="bf16"),
    "prec_fgmres_8": _c("prec", "fgmres", (40, 33, 21), 7, 14, precision="fp32"),
    "prec_fcg_units": _c("prec", "fcg", (2048, 1500, 1), 8, 8, precision="fp32"),   # more work units than blocks
    "prec_gcr_units": _c("prec", "gcr", (1500, 2048, 2), 4, 6, pc="chebyshev", precision="bf16"),
    "prec_fgmres_32": _c("prec", "fgmres", (40, 33, 21), 32, 32, pc="chebyshev", vel=ADV, precision="fp32"),
}


def problem(dims, seed):
    """Viscosities of contrast 2^10 and a right-hand side, exact in binary."""
    g = np.random.default_rng(seed)
    n = int(np.prod(dims))
    eta = np.ldexp(1.0 + g.integers(0, 1 << 20, n) / (1 << 20), g.integers(-5, 5, n).astype(np.int32))
    return eta, g.integers(-(1 << 20), 1 << 20, n) / float(1 << 30)


def solve_case(ctx, name):
    """[(x, iterations)] of the case."""
    from paper_1511_07226_gb300 import pfk
    c = CASES[name]
    prm = dict(method=c["method"], mmax=c["mmax"], maxit=c["maxit"], rtol=1e-14)
    dims = c["dims"] if isinstance(c["dims"], list) else [c["dims"]]
    probs = [problem(d, 7 + j) for j, d in enumerate(dims)]
    ops = [pfk.Operator.stencil(ctx, d, eta, c["vel"], storage=c["storage"]) for d, (eta, _) in zip(dims, probs)]
    if c["group"] == "grouped":
        xs, infos, _ = pfk.solve_grouped(ctx, ops, [b for _, b in probs], pc_kind=c["pc"], inner_iters=c["inner"],
                                         **prm)
        return [(x, i["iterations"]) for x, i in zip(xs, infos)]
    pc = pfk.Preconditioner(ctx, ops[0], c["pc"], inner_iters=c["inner"], precision=c.get("precision", "fp64"))
    x, info, _ = pfk.solve(ctx, ops[0], pc, probs[0][1], **prm)
    return [(x, info["iterations"])]


def summary(results):
    """Iterations and SAMPLES entries of every solution, exactly."""
    return [dict(iterations=int(it), x=[float(x[i]).hex() for i in np.linspace(0, x.size - 1, SAMPLES).astype(int)])
            for x, it in results]


if __name__ == "__main__":
    sys.path.insert(0, os.getcwd())
    from paper_1511_07226_gb300 import pfk
    out = {k: summary(solve_case(pfk.Context(0), k)) for k in CASES}
    json.dump(out, open(sys.argv[1], "w"), indent=0)
