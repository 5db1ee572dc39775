"""Workloads of the library as its users run them, through paper_1511_07226_gb300.pfk.

A case is one call (or, for serving, one burst of calls):

* ``apply``    Operator.apply: y = A x with the matrix-free stencil or assembled CSR;
* ``pc``       Preconditioner.apply: y = B(v), inner Jacobi-PCG or Chebyshev-Jacobi;
* ``solve``    pfk.solve: one system on the whole GPU, a fixed number of iterations;
* ``batched``  pfk.solve_batched: many 2D systems, one CTA each, host arrays;
* ``grouped``  pfk.solve_grouped: several 3D systems sharing the GPU, host arrays;
* ``serve``    Server.submit / poll: a burst of mixed 3D requests, host arrays.

Solves run a fixed number of iterations (maxit; the tolerance is out of reach):
the time per iteration is what a longer solve multiplies, and a count set by a
tolerance would move with rounding.  The iterates are compared before rounding
has been amplified: 16 to 48 iterations, contrasts up to 1e3.

Inputs are made on the GPU from the seed: a smooth random viscosity
eta = 10^(g) with clipped Gaussian g (correlation length 8 cells), right-hand
sides uniform in (-1, 1) scaled by h^2, and, where advection is on, a constant
velocity of global Peclet number 10.
"""
import math

import numpy as np
import torch

from paper_1511_07226_gb300 import pfk

RTOL = 1e-14          # out of reach within the iterations of a case
PECLET = 10.0


def _case(name, kind, nx, ny, nz=1, **kw):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, count=1, log_contrast=3.0, advect=False, csr=False,
             host=False, method="pipefcg", mmax=30, truncation="standard", maxit=40, pc="inner_pcg", inner=4,
             precision="fp64")
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a 2D operator on its own, latency only
        _case("apply_2d_64", "apply", 64, 64),
        # the largest operator: the advection-diffusion problem of the PIPEFGMRES workload
        _case("apply_3d_advect_256", "apply", 256, 256, 256, advect=True),
        # a preconditioner application on its own, ragged sides near the largest served request
        _case("pc_inner_pcg_ragged", "pc", 150, 141, 133),
        # the mixed-precision smoother: 8 Chebyshev sweeps, BF16 coefficients, FP32 vectors
        _case("pc_cheb_bf16_256", "pc", 256, 256, 256, advect=True, pc="chebyshev", inner=8, precision="bf16"),
        # a small latency-bound solve: assembled CSR, Jacobi, host arrays in and out
        _case("solve_csr_64", "solve", 64, 64, csr=True, host=True, pc="jacobi", maxit=48),
        # the headline: PIPEFCG(30) with 4 FP64 inner PCG iterations at 128^3
        _case("solve_pipefcg_128", "solve", 128, 128, 128),
        # its blocking baseline, on sides that are no multiple of anything
        _case("solve_fcg_ragged", "solve", 101, 97, 93, method="fcg"),
        # an ordinary mid-size solve by the residual-minimising method
        _case("solve_pipegcr_64", "solve", 64, 64, 64, method="pipegcr", maxit=20),
        # the largest solve: one restart cycle of PIPEFGMRES(30) at 256^3 with the BF16 smoother
        _case("solve_pipefgmres_256", "solve", 256, 256, 256, advect=True, log_contrast=2.0, method="pipefgmres",
              maxit=30, pc="chebyshev", inner=8, precision="bf16"),
        # many small 2D systems at once, FP32 inner PCG (sides nx/4 .. nx)
        _case("batched_2d", "batched", 160, 160, count=304, precision="fp32", maxit=12),
        # a launch full of small 3D systems (sides 5 nx/8 .. nx)
        _case("grouped_3d", "grouped", 40, 40, 40, count=57, maxit=24),
        # a burst of requests of mixed size and method: small ones grouped, larger ones on the workers
        _case("serve_burst", "serve", 80, 80, 80, count=8, maxit=20),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides3(rng, lo, hi):
    s = _log_uniform(rng, lo, hi)
    if rng.random() < 0.4:      # aligned cube
        s = max(8, s // 8 * 8)
        return s, s, s
    return tuple(min(hi, max(8, int(round(s * rng.uniform(0.85, 1.15))))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["apply", "pc", "solve", "solve", "solve", "batched", "grouped", "serve"])
    kw = dict(log_contrast=round(rng.uniform(1.0, 3.0), 3))
    if kind == "apply":
        if rng.random() < 0.3:
            dims = (_log_uniform(rng, 24, 2048), _log_uniform(rng, 24, 2048))
        else:
            dims = _sides3(rng, 24, 256)
            kw["advect"] = rng.random() < 0.5
        kw["csr"] = math.prod(dims) < 1 << 21 and rng.random() < 0.25
    elif kind == "pc":
        dims = _sides3(rng, 24, 256)
        kw["pc"] = rng.choice(["inner_pcg", "chebyshev"])
        kw["inner"] = rng.randint(4, 8)
        kw["precision"] = rng.choice(["fp64", "fp64", "fp32", "bf16"] if kw["pc"] == "chebyshev" else
                                     ["fp64", "fp64", "fp32"])
        kw["advect"] = kw["pc"] == "chebyshev" and rng.random() < 0.5
    elif kind == "solve":
        if rng.random() < 0.2:  # the small assembled problems
            s = _log_uniform(rng, 32, 128)
            dims = (s, max(16, int(s * rng.uniform(0.8, 1.2))))
            kw.update(csr=True, host=rng.random() < 0.5, pc="jacobi", maxit=rng.randint(32, 48),
                      method=rng.choice(["pipefcg", "fcg"]))
        else:
            kw["method"] = rng.choice(["pipefcg", "pipefcg", "fcg", "pipegcr", "pipefgmres", "gcr", "fgmres"])
            dims = _sides3(rng, 24, 160)
            kw["mmax"] = rng.choice([30, 30, 30, 16, 8])
            kw["maxit"] = (min(kw["mmax"], rng.randint(16, 30)) if "gmres" in kw["method"] else
                           rng.randint(16, 20) if kw["method"] == "pipegcr" or kw["mmax"] < 30 else
                           rng.randint(24, 40))
            kw["precision"] = "fp64"
            if kw["method"] in ("pipefcg", "fcg") and rng.random() < 0.3:
                kw.update(precision="fp32", maxit=rng.randint(16, 20))
            if "gmres" in kw["method"]:
                kw.update(pc="chebyshev", inner=8, advect=True, precision=rng.choice(["fp64", "bf16"]),
                          log_contrast=round(rng.uniform(1.0, 2.0), 3))
            elif kw["method"] in ("pipefcg", "fcg") and rng.random() < 0.25:
                kw["truncation"] = "restart"
    elif kind == "batched":
        s = rng.randint(96, 192)
        dims = (s, s)
        kw.update(count=rng.randint(64, 256), precision=rng.choice(["fp32", "fp64"]), maxit=rng.randint(8, 12))
    elif kind == "grouped":
        s = rng.randint(24, 56)
        dims = (s, s, s)
        kw.update(count=rng.randint(4, 60), method=rng.choice(["pipefcg", "pipefcg", "pipegcr", "pipefgmres"]),
                  maxit=rng.randint(16, 20))
        if kw["method"] == "pipefcg" and rng.random() < 0.4:
            kw["precision"] = "fp32"
    else:
        s = rng.randint(48, 96)
        dims = (s, s, s)
        kw.update(count=rng.randint(3, 10), maxit=rng.randint(16, 20))
    c = _case("", kind, *dims, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1 + int(seed))
    return g


def _problem(shape, log_contrast, gen):
    """Viscosity (shape z, y, x) of contrast 10^log_contrast, and b = h^2 f."""
    f = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    spec = torch.fft.rfftn(f)
    for ax, n in enumerate(shape):
        k = (torch.fft.rfftfreq if ax == len(shape) - 1 else torch.fft.fftfreq)(n, device="cuda", dtype=torch.float64)
        ell = min(8.0, n / 4.0)
        w = torch.exp(-(math.pi * ell * k) ** 2)
        spec = spec * w.reshape([-1 if a == ax else 1 for a in range(len(shape))])
    f = torch.fft.irfftn(spec, s=shape)
    f = ((f - f.mean()) / f.std()).clamp(-1.0, 1.0)
    eta = torch.pow(10.0, 0.5 * log_contrast * f)
    b = (torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) * 2.0 - 1.0) / shape[-1] ** 2
    return eta, b.reshape(-1)


def _velocity(case):
    return (PECLET / math.sqrt(3.0),) * 3 if case["advect"] else (0.0, 0.0, 0.0)


def _systems(case, seed):
    """[(shape, eta, b)] of the case, in order."""
    gen = _gen(seed)
    side, n = case["nx"], case["count"]
    if case["kind"] == "batched":
        sides = [side // 4 + (j * 7919) % (side - side // 4 + 1) for j in range(n)]
        shapes = [(s, s) for s in sides]
    elif case["kind"] == "grouped":
        sides = [5 * side // 8 + (j * 31) % (side - 5 * side // 8 + 1) for j in range(n)]
        shapes = [(s, s, s) for s in sides]
    elif case["kind"] == "serve":   # half of them small, half up to the full side
        sides = [max(16, side // 3) + (j // 2) % 9 if j % 2 else max(16, side - 5 * (j // 2)) for j in range(n)]
        shapes = [(s, s, s) for s in sides]
    else:
        shapes = [(case["nz"], case["ny"], case["nx"]) if case["nz"] > 1 else (case["ny"], case["nx"])]
    return [(s,) + _problem(s, case["log_contrast"], gen) for s in shapes]


def _serve_method(j):
    return ("pipefcg", "pipegcr", "pipefgmres")[j % 3]


def _dims(shape):
    return tuple(reversed(shape))


def _params(case):
    return dict(method=case["method"], mmax=case["mmax"], truncation=case["truncation"], maxit=case["maxit"],
                rtol=RTOL)


def prepare(case, seed):
    ctx = pfk.Context()
    st = dict(case=case, ctx=ctx)
    systems = _systems(case, seed)
    if case["kind"] == "serve":
        st["server"] = pfk.Server(ctx, workers=4)
        st["requests"] = [dict(dims=_dims(s), eta=e.reshape(-1).cpu().numpy(), b=b.cpu().numpy(),
                               method=_serve_method(j), mmax=case["mmax"], maxit=case["maxit"], rtol=RTOL,
                               pc_kind=case["pc"], inner_iters=case["inner"], precision=case["precision"])
                          for j, (s, e, b) in enumerate(systems)]
        return st
    st["ops"] = [pfk.Operator.stencil(ctx, _dims(s), e.reshape(-1), vel=_velocity(case),
                                      storage="csr" if case["csr"] else "matrix_free") for s, e, _ in systems]
    if case["kind"] in ("batched", "grouped"):
        st["bs"] = [b.cpu().numpy() for _, _, b in systems]
        return st
    st["b"] = systems[0][2].cpu().numpy() if case["host"] else systems[0][2]
    if case["kind"] != "apply":
        st["pc"] = pfk.Preconditioner(ctx, st["ops"][0], kind=case["pc"], inner_iters=case["inner"],
                                      precision=case["precision"])
    return st


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "apply":
        return state["ops"][0].apply(state["b"])
    if kind == "pc":
        return state["pc"].apply(state["b"])
    if kind == "solve":
        x, info, _ = pfk.solve(state["ctx"], state["ops"][0], state["pc"], state["b"], **_params(case))
        return x, info["iterations"]
    if kind in ("batched", "grouped"):
        kw = dict(pc_kind=case["pc"], inner_iters=case["inner"], precision=case["precision"], **_params(case))
        if kind == "batched":
            del kw["method"]
            xs, infos, _ = pfk.solve_batched(state["ctx"], state["ops"], state["bs"], **kw)
            return np.concatenate(xs), np.array([i["iterations"] for i in infos])
        xs, infos, _ = pfk.solve_grouped(state["ctx"], state["ops"], state["bs"], **kw)
        return xs, np.array([i["iterations"] for i in infos])
    srv = state["server"]
    tickets = [srv.submit(**r) for r in state["requests"]]
    done = [srv.poll(t) for t in tickets]
    return [x for x, _, _ in done], np.array([i["iterations"] for _, i, _ in done])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _op_work(case, n, ndim):
    """One operator application: bytes and flops (7- or 5-point, FP64)."""
    if case["csr"]:
        nnz = (2 * ndim + 1) * n
        return 12.0 * nnz + 20.0 * n, 2.0 * nnz
    adv = ndim if case["advect"] else 0
    return 8.0 * n * (ndim + 3), 2.0 * n * (2 * ndim + 1 + adv)


def _pc_work(case, n, ndim):
    """One preconditioner application: coefficients and v in, y out, and every
    inner iteration's vectors once."""
    if case["pc"] == "jacobi":
        return 24.0 * n, 1.0 * n
    v = 8.0 if case["precision"] == "fp64" else 4.0
    c = {"fp64": 8.0, "fp32": 4.0, "bf16": 2.0}[case["precision"]]
    coef = c * (ndim + 2) * n
    k = case["inner"]
    if case["pc"] == "inner_pcg":
        return 16.0 * n + k * (coef + 7.0 * v * n), 2.0 * n * k * (2 * ndim + 1 + 7)
    return 16.0 * n + (k - 1) * (coef + 6.0 * v * n), 2.0 * n * (k - 1) * (2 * ndim + 1 + 4)


def _iteration_work(method, nu, case, n, ndim):
    vec = 8.0 * n
    ob, of = _op_work(case, n, ndim)
    pb, pf = _pc_work(case, n, ndim)
    hist, other, fma = {"pipefcg": (4 * nu, 15, 5 * nu + 8), "fcg": (2 * nu, 10, 2 * nu + 4),
                        "pipegcr": (4 * nu, 17, 4 * nu + 9), "gcr": (2 * nu, 12, 2 * nu + 5),
                        "pipefgmres": (3 * nu, 7, 4 * nu + 5), "fgmres": (2 * nu, 6, 2 * nu + 3)}[method]
    nops = 2 if method == "gcr" else 1
    return vec * (hist + other) + nops * ob + pb, 2.0 * n * fma + nops * of + pf


def _solve_work(method, case, n, ndim):
    tb = tf = 0.0
    for i in range(case["maxit"]):
        nu = (i % case["mmax"]) + 1 if case["truncation"] == "restart" or "gmres" in method else min(i + 1, case["mmax"])
        b, f = _iteration_work(method, nu, case, n, ndim)
        tb, tf = tb + b, tf + f
    return tb, tf


def _shapes(case):
    side, n = case["nx"], case["count"]
    if case["kind"] == "batched":
        return [((side // 4 + (j * 7919) % (side - side // 4 + 1)) ** 2, 2) for j in range(n)]
    if case["kind"] == "grouped":
        return [((5 * side // 8 + (j * 31) % (side - 5 * side // 8 + 1)) ** 3, 3) for j in range(n)]
    if case["kind"] == "serve":
        return [((max(16, side // 3) + (j // 2) % 9 if j % 2 else max(16, side - 5 * (j // 2))) ** 3, 3)
                for j in range(n)]
    return [(case["nx"] * case["ny"] * case["nz"], 3 if case["nz"] > 1 else 2)]


def work(case):
    tb = tf = 0.0
    for j, (n, ndim) in enumerate(_shapes(case)):
        if case["kind"] == "apply":
            b, f = _op_work(case, n, ndim)
        elif case["kind"] == "pc":
            b, f = _pc_work(case, n, ndim)
        else:
            b, f = _solve_work(_serve_method(j) if case["kind"] == "serve" else case["method"], case, n, ndim)
        tb, tf = tb + b, tf + f
    return {"bytes": tb, "flops": tf}


# ---------------------------------------------------------------------------
# The same results in 64-bit torch
# ---------------------------------------------------------------------------

class _Stencil:
    """-div(eta grad u) with harmonic faces and Dirichlet ghosts, first-order
    upwind advection; `store` rounds the coefficients as a reduced-precision
    copy stores them."""

    def __init__(self, shape, eta, vel):
        self.shape, self.k, self.adv = shape, [], []
        nd = len(shape)
        d = torch.zeros(shape, dtype=torch.float64, device=eta.device)
        for a in range(nd - 1, -1, -1):
            n = shape[a]
            lo, hi = eta.narrow(a, 0, n - 1), eta.narrow(a, 1, n - 1)
            face = 2.0 * lo * hi / (lo + hi)
            first, last = 2.0 * eta.narrow(a, 0, 1), 2.0 * eta.narrow(a, n - 1, 1)
            d += torch.cat([first, face], a) + torch.cat([face, last], a)
            h = vel[nd - 1 - a] / shape[-1]
            d += abs(h)
            self.k.append((a, face))
            self.adv.append(abs(h))       # velocities here are >= 0: the upwind neighbour is at -1
        self.d, self.dinv = d, 1.0 / d

    def store(self, dtype):
        s = _Stencil.__new__(_Stencil)
        rnd = lambda t: t.float().to(dtype).double()  # noqa: E731
        s.shape, s.adv = self.shape, self.adv
        s.k = [(a, rnd(f)) for a, f in self.k]
        s.d, s.dinv = rnd(self.d), rnd(self.dinv)
        return s

    def __call__(self, u):
        u = u.reshape(self.shape)
        y = self.d * u
        for (a, face), h in zip(self.k, self.adv):
            n = self.shape[a]
            y.narrow(a, 0, n - 1).sub_(face * u.narrow(a, 1, n - 1))
            y.narrow(a, 1, n - 1).sub_((face + h) * u.narrow(a, 0, n - 1))
        return y.reshape(-1)

    def gershgorin(self):
        s = self.d.clone()
        for (a, face), h in zip(self.k, self.adv):
            n = self.shape[a]
            s.narrow(a, 0, n - 1).add_(face)
            s.narrow(a, 1, n - 1).add_(face + h)
        return float((s / self.d).max())


def _dot(a, b):
    return float(torch.dot(a, b))


def _pc_exact(case, A):
    dtype = {"fp64": torch.float64, "fp32": torch.float32, "bf16": torch.bfloat16}[case["precision"]]
    C = A if case["precision"] == "fp64" or case["pc"] == "jacobi" else A.store(dtype)
    dinv = C.dinv.reshape(-1)
    if case["pc"] == "jacobi":
        return lambda v: dinv * v
    k = case["inner"]
    if case["pc"] == "inner_pcg":
        def pcg(v):
            x, r = torch.zeros_like(v), v.clone()
            p = dinv * r
            gamma = _dot(p, r)
            for i in range(k):
                s = C(p)
                alpha = gamma / _dot(s, p)
                x = x + alpha * p
                if i + 1 < k:
                    r = r - alpha * s
                    u = dinv * r
                    gamma, old = _dot(u, r), gamma
                    p = u + (gamma / old) * p
            return x
        return pcg
    top = A.gershgorin()
    lo, hi = 0.1 * top, 1.1 * top

    def cheb(v):
        theta, delta = (hi + lo) / 2.0, (hi - lo) / 2.0
        rho = delta / theta
        r, x = v.clone(), torch.zeros_like(v)
        d = dinv * r / theta
        for j in range(k):
            x = x + d
            if j + 1 < k:
                r = r - C(d)
                new = 1.0 / (2.0 * theta / delta - rho)
                d = new * rho * d + (2.0 * new / delta) * (dinv * r)
                rho = new
        return x
    return cheb


def _window(i, case):
    return (i - 1) % case["mmax"] + 1 if case["truncation"] == "restart" else min(i, case["mmax"])


def _combine(base, beta, hist):
    out = base.clone()
    for k, c in beta.items():
        out.add_(hist[k], alpha=c)
    return out


def _cg_cr(method, case, A, B, b):
    """FCG, PIPEFCG, GCR and PIPEGCR (Alg. 2, 8, 9, 11) from x_0 = 0."""
    x, r = torch.zeros_like(b), b.clone()
    u = B(r)
    P, S, Q, Z = {0: u}, {0: A(u)}, {}, {}
    w = S[0]
    if method == "pipefcg":
        Q[0] = B(w)
        Z[0] = A(Q[0])
    if method == "pipegcr":
        Q[0] = B(w)
    cr = "gcr" in method
    eta = {0: _dot(S[0], S[0]) if cr else _dot(P[0], S[0])}
    alpha = (_dot(r, S[0]) if cr else _dot(u, r)) / eta[0]
    for i in range(1, case["maxit"] + 1):
        x = x + alpha * P[i - 1]
        if i == case["maxit"]:
            return x
        r = r - alpha * S[i - 1]
        if method in ("fcg", "gcr"):
            u = B(r)
            w = A(u) if cr else u
        else:
            u = u - alpha * Q[i - 1]
            w = w - alpha * Z[i - 1] if method == "pipefcg" else A(u)
        left = w if cr else u
        beta = {k: -_dot(left, S[k]) / eta[k] for k in range(i - _window(i, case), i)}
        P[i] = _combine(u, beta, P)
        if method in ("fcg", "gcr"):
            S[i] = A(P[i])
            eta[i] = _dot(S[i], S[i]) if cr else _dot(P[i], S[i])
            alpha = (_dot(r, S[i]) if cr else _dot(u, r)) / eta[i]
        else:
            m = u + B(w - r)
            S[i], Q[i] = _combine(w, beta, S), _combine(m, beta, Q)
            if method == "pipefcg":
                Z[i] = _combine(A(m), beta, Z)
            eta[i] = _dot(left, w) - sum(beta[k] ** 2 * eta[k] for k in beta)
            alpha = _dot(left, r) / eta[i]
        for h in (P, S, Q, Z):
            h.pop(i - case["mmax"] - 1, None)


def _gmres(method, case, A, B, b):
    """One cycle of FGMRES or PIPEFGMRES (Alg. 13, 15) from x_0 = 0."""
    m = case["maxit"]
    beta0 = float(torch.linalg.vector_norm(b))
    P = [b / beta0]
    U = [B(P[0])]
    H = np.zeros((m + 1, m))
    if method == "fgmres":
        for i in range(m):
            z = A(U[i])
            H[: i + 1, i] = [_dot(p, z) for p in P]
            for c, p in zip(H[: i + 1, i], P):
                z = z.sub(p, alpha=float(c))
            H[i + 1, i] = float(torch.linalg.vector_norm(z))
            if i + 1 < m:
                P.append(z / H[i + 1, i])
                U.append(B(P[-1]))
    else:
        v = P[0]
        for _ in range(10):     # the shift: 10 power iterations on A B
            y = A(B(v))
            sigma = float(torch.linalg.vector_norm(y))
            v = y / sigma
        Z = [A(U[0]) - sigma * P[0]]
        for i in range(m):
            h = np.array([_dot(p, Z[i]) for p in P])
            H[: i + 1, i] = h
            H[i, i] += sigma
            H[i + 1, i] = math.sqrt(_dot(Z[i], Z[i]) - float(np.sum(h * h)))
            if i + 1 < m:
                q = B(Z[i])
                new = [Z[i].clone(), q.clone(), A(q)]
                for j in range(i + 1):
                    new[0].sub_(P[j], alpha=float(h[j]))
                    new[1].sub_(U[j], alpha=float(h[j]))
                    new[2].sub_(Z[j], alpha=float(H[j, i]))
                for lst, vec in zip((P, U, Z), new):
                    lst.append(vec / H[i + 1, i])
    rhs = np.zeros(m + 1)
    rhs[0] = beta0
    y = np.linalg.lstsq(H, rhs, rcond=None)[0]
    x = torch.zeros_like(b)
    for c, u in zip(y, U):
        x.add_(u, alpha=float(c))
    return x


def _solution(method, case, shape, eta, b):
    A = _Stencil(shape, eta, _velocity(case))
    return (_gmres if "gmres" in method else _cg_cr)(method, case, A, _pc_exact(case, A), b)


def exact(case, seed):
    systems = _systems(case, seed)
    if case["kind"] in ("apply", "pc"):
        shape, eta, b = systems[0]
        A = _Stencil(shape, eta, _velocity(case))
        return A(b) if case["kind"] == "apply" else _pc_exact(case, A)(b)
    xs = [_solution(_serve_method(j) if case["kind"] == "serve" else case["method"], case, *s)
          for j, s in enumerate(systems)]
    if case["kind"] == "solve":
        return xs[0].cpu().numpy() if case["host"] else xs[0], None
    xs = [x.cpu().numpy() for x in xs]
    return np.concatenate(xs) if case["kind"] == "batched" else xs, None
