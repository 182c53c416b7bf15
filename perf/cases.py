"""The pricing library's performance cases: what its users run, over the sizes they run it at.

A user prices options (one at a time, in a batch, with a gradient), applies the jump operator or
one fixed-point iteration of their own time loop, or runs the paper's price-space scheme.  Each
case is one such call through the package's public entry points; parameters follow the ranges of
paper_2511_02700_gb300/workloads.py (``batch_draw``, ``convergence_sweep``, the paper's Table 2).

FP32-bulk results are kept in FP32, the precision that mode gives; FP64 results in FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_02700_gb300 import binding as B
from paper_2511_02700_gb300.workloads import PAPER_SETS

DEV = "cuda"
STRIKE_NODE = 100.0            # S0 of both assets: the centre of the log grid
HALF_WIDTH = 2.5


# ------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the jump sum with given weights in a process that may not allocate: the smallest call,
        # bound by its launches
        dict(name="static_fp64_64", kind="static", n=64),
        # one application of the jump operator inside a user's own scheme, both precisions
        dict(name="jump_fp32_512", kind="jump", n=512, precision="fp32", alpha=0.5, payoff=0),
        dict(name="jump_fp64_1024", kind="jump", n=1024, precision="fp64", alpha=0.25, payoff=1),
        # one fixed-point iteration at the largest grid: the kernels the big solve spends its time in
        dict(name="iteration_fp32_4096", kind="iteration", n=4096, precision="fp32", alpha=0.5),
        # an ordinary FP64 quote: model in, price surface out (128^2 grid, 32 steps, tol 1e-10)
        dict(name="price_fp64_128", kind="price", n=128, steps=32, precision="fp64", alpha=0.25, tol=1e-10,
             maturity=1.0, payoff=0, sl_order=3),
        # the fast mode's ordinary quote (convergence sweep: steps N/4, tol 1e-8), and the same in FP64
        dict(name="price_fp32_512", kind="price", n=512, steps=128, precision="fp32", alpha=0.5, tol=1e-8,
             maturity=1.0, payoff=0, sl_order=3),
        dict(name="price_fp64_512", kind="price", n=512, steps=128, precision="fp64", alpha=0.5, tol=1e-8,
             maturity=1.0, payoff=1, sl_order=3),
        # the large solve (8192^2 transforms, time step 1/1024, tol 1e-7) over its first 64 steps
        dict(name="price_fp32_4096", kind="price", n=4096, steps=64, precision="fp32", alpha=0.5, tol=1e-7,
             maturity=0.0625, payoff=0, sl_order=3),
        # a book of independent options of mixed sizes, models, strikes and maturities
        dict(name="batch_fp32_48", kind="batch", count=48, tol=1e-8),
        # price and gradient with respect to the six model parameters (forward, checkpoints, adjoint)
        dict(name="adjoint_fp64_256", kind="adjoint", n=256, steps=64, alpha=0.25, tol=1e-10, interval=16),
        # the paper's scheme on its non-uniform price grid: the operator, and a whole pricing
        dict(name="space_jump_fp64_320", kind="space_jump", set="VG1", nx=320, precision="fp64"),
        dict(name="space_price_fp64_150", kind="space_price", set="NIG1", nx=150, steps=75, precision="fp64",
             tol=1e-7),
    ]


def draw(rng):
    def pow2(lo, hi):
        return 1 << rng.randint(lo, hi)

    alpha = round(rng.uniform(0.1, 0.6), 3)
    prec = rng.choice(("fp32", "fp64"))
    kind = rng.choice(("static", "jump", "jump", "iteration", "iteration", "price", "price", "price", "price", "batch",
                       "adjoint", "space_jump", "space_price"))
    if kind == "static":
        return dict(kind=kind, n=pow2(3, 8), scale=alpha)
    if kind == "jump":
        return dict(kind=kind, n=pow2(5, 12 if prec == "fp32" else 11), precision=prec, alpha=alpha,
                    payoff=rng.randint(0, 2))
    if kind == "iteration":
        return dict(kind=kind, n=pow2(5, 12 if prec == "fp32" else 11), precision=prec, alpha=alpha)
    if kind == "price":
        n = pow2(4, 11 if prec == "fp32" else 9)
        steps = max(4, int(n * rng.uniform(0.1, 0.25)))
        return dict(kind=kind, n=n, steps=steps, precision=prec, alpha=alpha, maturity=round(rng.uniform(0.1, 1.0), 3),
                    tol=rng.choice((1e-7, 1e-8)) if prec == "fp32" else rng.choice((1e-8, 1e-10)),
                    payoff=rng.randint(0, 2), sl_order=rng.choice((1, 3, 3)))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 48), tol=rng.choice((1e-7, 1e-8)))
    if kind == "adjoint":
        n = pow2(5, 8)
        return dict(kind=kind, n=n, steps=max(4, int(n * rng.uniform(0.1, 0.25))), alpha=round(rng.uniform(0.1, 0.45), 3),
                    tol=1e-10, interval=rng.choice((4, 8, 16)))
    which = rng.choice(("VG1", "NIG1", "NIG1"))
    if kind == "space_jump":
        return dict(kind=kind, set=which, nx=int(math.exp(rng.uniform(math.log(24), math.log(200)))),
                    precision="fp64")
    nx = int(math.exp(rng.uniform(math.log(24), math.log(150))))
    return dict(kind=kind, set=which, nx=nx, steps=max(4, nx // 2), precision="fp64", tol=1e-7)


# ------------------------------------------------------------------------- inputs (from the seed)
def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _workload(rng, alpha):
    """(alpha, kappa, beta, sigma, corr, r) around the repository's workloads."""
    return dict(alpha=alpha, kappa=float(rng.uniform(0.3, 0.6)),
                beta=(float(rng.uniform(-0.15, 0.0)), float(rng.uniform(-0.1, 0.05))),
                sigma=(float(rng.uniform(0.15, 0.25)), float(rng.uniform(0.2, 0.3))),
                corr=float(rng.uniform(-0.2, 0.5)), r=0.03)


def _precision(case):
    return B.PIDE2D_FP64 if case["precision"] == "fp64" else B.PIDE2D_FP32_BULK


def _kept(case, t):
    """Results as a caller of that precision keeps them."""
    return t if case["precision"] == "fp64" else t.float()


def _field(n, seed):
    """A price-like field with node-to-node variation: values in [0, 100] on (n+1)^2 nodes."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    return 100.0 * torch.rand((n + 1, n + 1), generator=g, dtype=torch.float64, device=DEV)


def _surface(x, K, seed):
    """A smooth price surface of a put on the average over the price grid x."""
    rng = _rng(seed + 1)
    t, width = torch.as_tensor(x, device=DEV), K * float(rng.uniform(0.05, 0.15))
    w = float(rng.uniform(0.4, 0.6))
    return width * torch.nn.functional.softplus((K - w * t[None, :] - (1.0 - w) * t[:, None]) / width)


def _price_inputs(case, seed):
    rng = _rng(seed)
    return _workload(rng, case["alpha"]), float(rng.uniform(90.0, 110.0))


def _batch_inputs(case, seed):
    """The parameter draws of a book (the ranges of workloads.batch_draw)."""
    rng = _rng(seed)
    jobs = []
    for _ in range(case["count"]):
        w = dict(alpha=float(rng.uniform(0.1, 0.45)), kappa=float(rng.uniform(0.2, 1.0)),
                 sigma=(float(rng.uniform(0.1, 0.4)), float(rng.uniform(0.1, 0.4))),
                 corr=float(rng.uniform(-0.6, 0.6)),
                 beta=(float(rng.uniform(-0.2, 0.2)), float(rng.uniform(-0.2, 0.2))), r=0.03)
        n = int(rng.choice([128, 256, 512]))
        jobs.append((w, n, n // 4, float(rng.uniform(80.0, 120.0)), float(rng.uniform(0.1, 2.0))))
    return jobs


def _space_inputs(case, seed):
    """The paper's set with its strike moved: the grid scales with it."""
    p = PAPER_SETS[case["set"]]
    K = float(_rng(seed).uniform(80.0, 120.0))
    x, n_z, h_z, ny_minus, ny_plus = B.price_sinh_grid(case["nx"], K, p.x_max_over_k * K, p.z_max_iii)
    return p, K, x, n_z, h_z, ny_minus, ny_plus


def _static_inputs(case, seed):
    """Weights as a jump measure's: positive, peaked at the origin, decaying."""
    n, rng = case["n"], _rng(seed)
    z = (torch.arange(-(n // 2), n // 2, dtype=torch.float64, device=DEV) + 0.5) * (2 * HALF_WIDTH / n)
    q = z[None, :] ** 2 * rng.uniform(10.0, 30.0) + z[:, None] ** 2 * rng.uniform(10.0, 30.0)
    omega = torch.exp(-torch.sqrt(q)) / (0.01 + q) * (2 * HALF_WIDTH / n) ** 2
    return omega, _field(n, seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "static":
        omega, U = _static_inputs(case, seed)
        return dict(case=case, omega=omega, U=U, out=torch.zeros_like(U))
    if kind in ("jump", "iteration"):
        w, strike = _price_inputs(case, seed)
        model = B.model_from_subordinated_bm(w["alpha"], w["kappa"], w["beta"], w["sigma"], w["corr"], w["r"])
        s = B.Solver(B.make_grid(case["n"], _precision(case)), model,
                     B.make_contract(case.get("payoff", 0), strike, 1.0), 64, tol=1e-8)
        U = _field(case["n"], seed)
        if kind == "iteration":
            U = U / 50.0 - 1.0
        return dict(case=case, solver=s, U=U)
    if kind == "price":
        w, strike = _price_inputs(case, seed)
        model = B.model_from_subordinated_bm(w["alpha"], w["kappa"], w["beta"], w["sigma"], w["corr"], w["r"])
        return dict(case=case, grid=B.make_grid(case["n"], _precision(case), case["sl_order"]), model=model,
                    contract=B.make_contract(case["payoff"], strike, case["maturity"]))
    if kind == "batch":
        jobs = [B.make_job(B.make_grid(n, B.PIDE2D_FP32_BULK),
                           B.model_from_subordinated_bm(w["alpha"], w["kappa"], w["beta"], w["sigma"], w["corr"],
                                                        w["r"]),
                           B.make_contract(B.PIDE2D_PUT_AVG, K, T), steps, tol=case["tol"])
                for w, n, steps, K, T in _batch_inputs(case, seed)]
        return dict(case=case, jobs=jobs)
    if kind == "adjoint":
        w, strike = _price_inputs(case, seed)
        params = torch.tensor([w["sigma"][0], w["sigma"][1], w["corr"], w["kappa"], w["beta"][0], w["beta"][1]],
                              dtype=torch.float64, requires_grad=True)
        return dict(case=case, params=params, w=w, grid=B.make_grid(case["n"], B.PIDE2D_FP64),
                    contract=B.make_contract(B.PIDE2D_PUT_AVG, strike, 1.0), price=B.price_function())
    p, K, x, n_z, h_z, ny_minus, ny_plus = _space_inputs(case, seed)
    model = B.make_model(p.alpha, p.delta, p.lam, p.eta, p.rho, p.r)
    op = B.PriceJump(x, n_z, h_z, ny_minus, ny_plus, model, precision=_precision(case))
    st = dict(case=case, op=op, contract=B.make_contract(B.PIDE2D_PUT_AVG, K, p.maturity))
    if kind == "space_jump":
        st["V"] = _surface(x, K, seed)
    return st


# --------------------------------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "static":
        B.pide2d_jump_static(case["n"], st["omega"].data_ptr(), st["U"].data_ptr(), st["out"].data_ptr())
        return st["out"]
    if kind == "jump":
        return _kept(case, st["solver"].apply_jump(st["U"], 0.5))
    if kind == "iteration":
        delta, bdelta, stop = st["solver"].iteration_probe(st["U"], 1.0 / 1024, 0.5)
        return dict(delta=_kept(case, delta), bdelta=_kept(case, bdelta), stop=stop)
    if kind == "price":
        s = B.Solver(st["grid"], st["model"], st["contract"], case["steps"], tol=case["tol"])
        price, V, _, _ = s.solve(values=True)
        s.close()
        return dict(price=price, values=_kept(case, V))
    if kind == "batch":
        prices, statuses, _ = B.solve_batch(st["jobs"])
        return dict(prices=torch.tensor(prices, dtype=torch.float32), statuses=torch.tensor(statuses))
    if kind == "adjoint":
        p = st["params"]
        p.grad = None
        price = st["price"].apply(p, case["alpha"], st["w"]["r"], st["grid"], st["contract"], case["steps"], 0.5,
                                  case["tol"], case["interval"])
        price.backward()
        return dict(price=price.detach(), grad=p.grad)
    if kind == "space_jump":
        return _kept(case, st["op"].apply(st["V"]))
    V, _, _ = st["op"].solve(st["contract"], case["steps"], tol=case["tol"])
    return V


# ------------------------------------------------------------- what a pass cannot do without
def _sweep_flops(P):
    """Real 2D transform of P x P points forward and back (2.5 P^2 log2 P^2 each)."""
    return 2 * 2.5 * P * P * 2 * math.log2(P)


def work(case):
    kind = case["kind"]
    if kind == "static":
        n = case["n"]
        return dict(bytes=8.0 * (n * n + 2 * (n + 1) ** 2), flops=1.5 * _sweep_flops(2 * n))
    if kind in ("space_jump", "space_price"):
        # fields in and out; a transform as long as the kept lattice needs
        nodes = float((case["nx"] + 1) ** 2)
        lattice = 8 * case["nx"]
        sweeps = 1 if kind == "space_jump" else 2 * case["steps"]
        return dict(bytes=16.0 * nodes * sweeps, flops=_sweep_flops(lattice) * sweeps)
    if kind == "batch":
        shapes = [(n, n // 4) for n in (128, 256, 512)]
        each = [dict(kind="price", n=n, steps=s, precision="fp32") for n, s in shapes]
        parts = [work(dict(e, tol=0)) for e in each]
        return {k: case["count"] * sum(p[k] for p in parts) / len(parts) for k in ("bytes", "flops")}
    n = case["n"]
    cells = float((n + 1) ** 2)
    elem = 8.0
    if kind == "jump":
        return dict(bytes=2 * elem * cells + 8.0 * n * n, flops=_sweep_flops(2 * n))
    if kind == "iteration":
        return dict(bytes=3 * elem * cells + 8.0 * n * n, flops=1.5 * _sweep_flops(2 * n))
    # a time step reads and writes the value field and applies the jump operator at least twice
    # (the start of the iteration, one iteration), each with its weights and one field in and out
    sweeps = 2 * case["steps"] * (3 if kind == "adjoint" else 1)
    return dict(bytes=sweeps * (2 * elem * cells + 8.0 * n * n), flops=sweeps * 1.25 * _sweep_flops(2 * n))


# ------------------------------------------------- the same in 64 bits, by plain torch and numpy
MID = (-1.0 / 16, 9.0 / 16, 9.0 / 16, -1.0 / 16)     # cubic Lagrange at a cell's midpoint


def _t(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device=DEV)


def _model(w):
    """(alpha, delta, lambda, eta, rho, r) of a unit-mean tempered-stable subordinator of variance kappa."""
    a = w["alpha"]
    lam = (1.0 - a) / w["kappa"]
    s1, s2 = w["sigma"]
    return dict(alpha=a, delta=lam ** (1.0 - a) / math.gamma(1.0 - a), lam=lam, eta=w["beta"],
                rho=(s1 * s1, w["corr"] * s1 * s2, s2 * s2), r=w["r"])


def _log_scaled_bessel(nu, x):
    """ln(e^x K_nu(x)): the trapezoidal rule on K_nu(x) = int_0^inf e^{-x cosh t} cosh(nu t) dt."""
    lo = float(x.min())
    step = 0.08
    out = torch.full_like(x, 0.5 * step)             # t = 0: the integrand of e^x K_nu is 1
    t = step
    while True:
        c = 2.0 * math.sinh(0.5 * t) ** 2             # cosh t - 1
        if lo * c > 60.0 + nu * t:
            return torch.log(out)
        out += (step * math.cosh(nu * t)) * torch.exp(-c * x)
        t += step


def _density(m, z1, z2):
    """The NTS Levy density delta/pi sqrt(c^(2 nu)/det rho) K_nu(c |z|) |z|^-nu e^<eta, z>, nu = 1 + alpha,
    in the norm of rho^-1, c = sqrt(|eta|^2 + 2 lambda)."""
    r11, r12, r22 = m["rho"]
    det = r11 * r22 - r12 * r12
    i11, i12, i22 = r22 / det, -r12 / det, r11 / det
    b1 = i11 * m["eta"][0] + i12 * m["eta"][1]
    b2 = i12 * m["eta"][0] + i22 * m["eta"][1]
    c = math.sqrt(m["eta"][0] * b1 + m["eta"][1] * b2 + 2.0 * m["lam"])
    nu = 1.0 + m["alpha"]
    z1, z2 = torch.broadcast_tensors(z1, z2)
    zn = torch.sqrt(i11 * z1 * z1 + 2.0 * i12 * z1 * z2 + i22 * z2 * z2)
    x = c * zn
    tiny = x < 1e-6                                   # K_nu(x) -> Gamma(nu) 2^(nu - 1) x^-nu
    lk = _log_scaled_bessel(nu, torch.where(tiny, torch.ones_like(x), x)) - x
    lk = torch.where(tiny, math.lgamma(nu) + (nu - 1.0) * math.log(2.0) - nu * torch.log(x), lk)
    const = math.log(m["delta"] / math.pi) + nu * math.log(c) - 0.5 * math.log(det)
    return torch.exp(const + lk - nu * torch.log(zn) + b1 * z1 + b2 * z2)


def _quadrature(m, nz, h):
    """Weights [l2, l1] on 2 nz cells of width h per axis (0 for |z| <= 2h; cell integrals of |z|^2 l over the
    middle of the range; l(z) h^2 beyond), r_w, kappa_w, the small-jump covariance (a11, a12, a22)."""
    l = np.arange(-nz, nz) + 0.5
    z = _t(l * h)
    inf = np.maximum(np.abs(l)[None, :], np.abs(l)[:, None])
    mid = (inf > 2) & (inf <= int(math.ceil(math.sqrt(0.1) * nz - 0.5)))
    om = torch.zeros((2 * nz, 2 * nz), dtype=torch.float64, device=DEV)
    for r in range(0, 2 * nz, 1024):
        om[r:r + 1024] = _density(m, z[None, :], z[r:r + 1024, None]) * (h * h)
    om *= torch.as_tensor(inf > 2, device=DEV)
    i2, i1 = (torch.as_tensor(v, device=DEV) for v in np.nonzero(mid))
    c1, c2 = z[i1], z[i2]
    gx, gw = np.polynomial.legendre.leggauss(12)
    cell = torch.zeros_like(c1)
    for a in range(12):
        for b in range(12):
            z1, z2 = c1 + 0.5 * h * gx[a], c2 + 0.5 * h * gx[b]
            cell += (0.25 * h * h * gw[a] * gw[b]) * (z1 * z1 + z2 * z2) * _density(m, z1, z2)
    om[i2, i1] = cell / (c1 * c1 + c2 * c2)
    # int over |z|_inf <= 2h of z z^T l(z): four triangles with their apex at 0, tanh-sinh along the rays
    u = np.arange(-420, 421) / 100.0
    s = 0.5 * math.pi * np.sinh(u)
    rho = 2.0 * h * 1.0 / (1.0 + np.exp(-2.0 * s))
    wr = 2.0 * h * 0.01 * 0.5 * math.pi * np.cosh(u) * 0.5 / np.cosh(s) ** 2
    keep = rho > 1e-100
    rho, wr = _t(rho[keep])[:, None], _t(wr[keep])[:, None]
    gx, gw = np.polynomial.legendre.leggauss(64)
    t, wt = _t(gx)[None, :], _t(gw)[None, :]
    a = [0.0, 0.0, 0.0]
    for d1, d2 in ((torch.ones_like(t), t), (-torch.ones_like(t), t), (t, torch.ones_like(t)), (t, -torch.ones_like(t))):
        f = wr * wt * rho ** 3 * _density(m, rho * d1, rho * d2)
        a = [v + float((f * q).sum()) for v, q in zip(a, (d1 * d1, d1 * d2, d2 * d2))]
    e = torch.expm1(z)
    kappa = (m["r"] - float((om * e[None, :]).sum()), m["r"] - float((om * e[:, None]).sum()))
    return om, m["r"] + float(om.sum()), kappa, a


def _correlate(om_hat, A, P):
    return torch.fft.irfft2(om_hat * torch.fft.rfft2(A, s=(P, P)), s=(P, P))


class _LogScheme:
    """The semi-Lagrangian theta scheme on the uniform log grid ln S0 +- 2.5, each step's equation solved until
    the increment no longer matters in 64 bits."""

    def __init__(self, m, n, payoff, strike):
        self.n, self.r, self.payoff, self.strike = n, m["r"], payoff, strike
        self.h = 2 * HALF_WIDTH / n
        om, self.rw, kappa, self.a = _quadrature(m, n // 2, self.h)
        self._set_weights(om)
        self.b = (kappa[0] - 0.5 * self.a[0], kappa[1] - 0.5 * self.a[2])
        k = np.arange(1, n)
        self.eig = _t((2.0 - 2.0 * np.cos(np.pi * k / n)) / self.h ** 2)

    def _set_weights(self, om):
        P = 2 * self.n
        self.om_hat = torch.conj(torch.fft.rfft2(om, s=(P, P)))

    def far(self, tau, lo, hi):
        """The payoff with the strike discounted, at nodes lo..hi of both axes."""
        s = math.log(STRIKE_NODE) - HALF_WIDTH + torch.arange(lo, hi + 1, dtype=torch.float64, device=DEV) * self.h
        e, K = torch.exp(s), self.strike * math.exp(-self.r * tau)
        avg = 0.5 * (e[None, :] + e[:, None])
        return torch.clamp((K - avg, avg - K, K - e[None, :] + 0.0 * avg)[self.payoff], min=0.0)

    def jump(self, inner, tau, far=True):
        """The jump sum at the interior nodes, `inner` there and the far field (or 0) outside."""
        n = self.n
        nz = n // 2
        U = self.far(tau, -nz - 1, n + nz) if far else torch.zeros((2 * n + 2, 2 * n + 2), dtype=torch.float64, device=DEV)
        U[nz + 2:nz + 1 + n, nz + 2:nz + 1 + n] = inner
        k = U.shape[0] - 3
        A = sum(MID[q] * U[:, q:k + q] for q in range(4))
        A = sum(MID[q] * A[q:k + q, :] for q in range(4))
        return _correlate(self.om_hat, A, 2 * n)[1:n, 1:n]

    def diffuse(self, V):
        a, h2 = self.a, self.h ** 2
        c = V[1:-1, 1:-1]
        return (0.5 * a[0] * (V[1:-1, 2:] - 2 * c + V[1:-1, :-2]) + 0.5 * a[2] * (V[2:, 1:-1] - 2 * c + V[:-2, 1:-1])
                + 0.25 * a[1] * (V[2:, 2:] - V[:-2, 2:] - V[2:, :-2] + V[:-2, :-2])) / h2

    def _dst(self, X, dim):
        z = torch.zeros_like(X.narrow(dim, 0, 1))
        return -torch.fft.rfft(torch.cat((z, X, z, -X.flip(dim)), dim), dim=dim).imag.narrow(dim, 1, self.n - 1)

    def solve_nonmixed(self, R, ht, theta):
        lam = 1.0 + ht * theta * (self.rw + 0.5 * self.a[0] * self.eig[None, :] + 0.5 * self.a[2] * self.eig[:, None])
        X = self._dst(self._dst(R, 0), 1) / lam
        return self._dst(self._dst(X, 0), 1) / (2.0 * self.n) ** 2

    def initial(self):
        """The payoff, averaged over the cells that its kink crosses."""
        n, h, K = self.n, self.h, self.strike
        V = self.far(0.0, 0, n)
        s = math.log(STRIKE_NODE) - HALF_WIDTH + np.arange(n + 1) * h
        if self.payoff == 2:
            m1 = np.nonzero((np.exp(s - 0.5 * h) < K) & (K < np.exp(s + 0.5 * h)))[0]
            for i in m1[(m1 > 0) & (m1 < n)]:
                a, up = s[i] - 0.5 * h, math.log(K)
                V[1:n, i] = (K * (up - a) - (math.exp(up) - math.exp(a))) / h
            return V
        lo, hi = np.exp(s - 0.5 * h), np.exp(s + 0.5 * h)
        m2, m1 = np.nonzero((lo[:, None] + lo[None, :] < 2 * K) & (hi[:, None] + hi[None, :] > 2 * K))
        ok = (m1 > 0) & (m1 < n) & (m2 > 0) & (m2 < n)
        m1, m2 = m1[ok], m2[ok]
        a1, a2 = s[m1] - 0.5 * h, s[m2] - 0.5 * h
        gx, gw = np.polynomial.legendre.leggauss(20)

        def cross(edge):                              # where the kink meets a vertical edge of the cell
            q = 2 * K - np.exp(edge)
            return np.clip(np.where(q > 0, np.log(np.where(q > 0, q, 1.0)), -np.inf), a2, a2 + h)

        cuts = np.sort(np.stack((a2, cross(a1), cross(a1 + h), a2 + h)), axis=0)
        total = np.zeros_like(a1)
        for p in range(3):
            half = 0.5 * (cuts[p + 1] - cuts[p])
            for g, w in zip(gx, gw):
                c = K - 0.5 * np.exp(cuts[p] + half * (1.0 + g))
                # inner integral of (c - e^s / 2)^+ over the cell's s1 range, and of the call's by parity
                top = np.clip(np.where(c > 0, np.log(np.where(c > 0, 2 * c, 1.0)), -np.inf), a1, a1 + h)
                put = c * (top - a1) - 0.5 * (np.exp(top) - np.exp(a1))
                put = np.where(c > 0, put, 0.0)
                if self.payoff == 1:
                    put = put - c * h + 0.5 * (np.exp(a1 + h) - np.exp(a1))
                total += w * half * put
        V[torch.as_tensor(m2, device=DEV), torch.as_tensor(m1, device=DEV)] = _t(total / (h * h))
        return V

    def theta_step(self, V, BV, start, tau0, ht, theta, order):
        n, tau = self.n, tau0 + ht
        Vi = V[1:-1, 1:-1]
        pad = 8 + n // 4
        Z = self.far(tau0, -pad, n + pad)
        Z[pad + 1:pad + n, pad + 1:pad + n] = Vi + ht * (1 - theta) * (self.diffuse(V) - self.rw * Vi + BV)
        taps = []
        for b in self.b:
            q = b * ht / self.h
            o = math.floor(q)
            f = q - o
            taps.append((o, (1 - f, f)) if order == 1 else
                        (o - 1, (-f * (f - 1) * (f - 2) / 6, (f + 1) * (f - 1) * (f - 2) / 2,
                                 -(f + 1) * f * (f - 2) / 2, (f + 1) * f * (f - 1) / 6)))
        (o1, w1), (o2, w2) = taps
        W = sum(wb * wa * Z[pad + 1 + o2 + j:pad + o2 + j + n, pad + 1 + o1 + i:pad + o1 + i + n]
                for j, wb in enumerate(w2) for i, wa in enumerate(w1))
        Y = self.far(tau, 0, n)
        Y[1:-1, 1:-1] = start
        BY = self.jump(start, tau)
        last = math.inf
        for _ in range(60):
            Yi = Y[1:-1, 1:-1]
            D = self.solve_nonmixed(W - Yi + ht * theta * (BY - self.rw * Yi + self.diffuse(Y)), ht, theta)
            Yi += D
            size = float(D.abs().max()) / self.strike
            BY = BY + self.jump(D, tau, far=False)
            if size < 1e-12 or size >= 0.7 * last and size < 1e-9:
                break
            last = size
        return Y, BY

    def solve(self, steps, maturity, order=3):
        ht = maturity / steps
        V0 = self.initial()
        V, BV = V0, self.jump(V0[1:-1, 1:-1], 0.0)
        for j in range(4):
            V, BV = self.theta_step(V, BV, V[1:-1, 1:-1], j * ht / 4, ht / 4, 1.0, order)
        hist = [V, V0]
        for k in range(1, steps):
            c = ((1,), (2, -1), (3, -3, 1), (4, -6, 4, -1))[len(hist) - 1]
            start = sum(q * v[1:-1, 1:-1] for q, v in zip(c, hist))
            V, BV = self.theta_step(V, BV, start, k * ht, ht, 0.5, order)
            hist = [V] + hist[:3]
        return V


def _lagrange(nodes, targets, outside):
    """Dense interpolation matrix: cubic Lagrange on the four nodes around each target (shifted inside at the
    ends); beyond the nodes linear, or an empty row above the last node with outside = 'zero'."""
    n = nodes.size
    M = np.zeros((targets.size, n))
    for i, t in enumerate(targets):
        if t > nodes[-1] and outside == "zero":
            continue
        if t > nodes[-1] or t < nodes[0]:
            j = 0 if t < nodes[0] else n - 2
            d = nodes[j + 1] - nodes[j]
            M[i, j], M[i, j + 1] = (nodes[j + 1] - t) / d, (t - nodes[j]) / d
            continue
        k = min(max(int(np.searchsorted(nodes, t, side="right")) - 1, 0), n - 2)
        s = min(max(k - 1, 0), n - 4)
        for q in range(s, s + 4):
            M[i, q] = np.prod([(t - nodes[r]) / (nodes[q] - nodes[r]) for r in range(s, s + 4) if r != q])
    return _t(M)


class _PriceScheme:
    """The paper's scheme on its price grid: B = T_out C T_in, D on the non-uniform nodes, theta steps."""

    def __init__(self, case, seed):
        p, K, x, n_z, h_z, nm, npl = _space_inputs(case, seed)
        m = dict(alpha=p.alpha, delta=p.delta, lam=p.lam, eta=p.eta, rho=p.rho, r=p.r)
        om, self.rw, self.kappa, self.a = _quadrature(m, n_z, h_z)
        self.x, self.K, self.maturity = x, K, p.maturity
        self.t_in = _lagrange(x, np.exp((np.arange(-n_z - nm, n_z + npl) + 0.5) * h_z), "zero")
        self.t_out = _lagrange(np.exp(np.arange(-nm, npl + 1) * h_z), x, "linear")
        self.P = max(self.t_in.shape[0], 4 * n_z)
        self.om_hat = torch.conj(torch.fft.rfft2(om, s=(self.P, self.P)))
        d = np.diff(x)
        D1, D2 = np.zeros((x.size, x.size)), np.zeros((x.size, x.size))
        for i in range(1, x.size - 1):
            l, r = d[i - 1], d[i]
            D1[i, i - 1:i + 2] = -r / (l * (l + r)), (r - l) / (l * r), l / (r * (l + r))
            D2[i, i - 1:i + 2] = 2 / (l * (l + r)), -2 / (l * r), 2 / (r * (l + r))
        D1[-1, -2:] = -1 / d[-1], 1 / d[-1]
        self.D1, self.D2 = _t(x[:, None] * D1), _t((x * x)[:, None] * D2)
        self._tables = {}

    def jump(self, V):
        k = self.t_out.shape[1]
        return self.t_out @ _correlate(self.om_hat, self.t_in @ V @ self.t_in.T, self.P)[:k, :k] @ self.t_out.T

    def diffuse(self, V):
        a = self.a
        return 0.5 * a[0] * V @ self.D2.T + a[1] * self.D1 @ V @ self.D1.T + 0.5 * a[2] * self.D2 @ V

    def solve(self, steps, theta=0.5):
        x, K = self.x, self.K
        mid = 0.5 * (x[1:] + x[:-1])
        lo, hi = np.concatenate(([-mid[0]], mid)), np.concatenate((mid, [2 * x[-1] - mid[-1]]))
        A1, A2, B1, B2 = lo[None, :], lo[:, None], hi[None, :], hi[:, None]

        def third(t):
            return np.maximum(t, 0.0) ** 3 / 6.0

        avg = 4.0 * (third(K - A1 / 2 - A2 / 2) - third(K - A1 / 2 - B2 / 2) - third(K - B1 / 2 - A2 / 2)
                     + third(K - B1 / 2 - B2 / 2)) / ((B1 - A1) * (B2 - A2))
        kink = (A1 + A2 < 2 * K) & (B1 + B2 > 2 * K)
        V = _t(np.where(kink, avg, np.maximum(K - 0.5 * (x[None, :] + x[:, None]), 0.0)))
        BV, hist, ht = self.jump(V), [V], self.maturity / steps
        for j in range(4):
            V, BV = self._step(V, BV, V, ht / 4, 1.0)
        hist = [V] + hist
        for _ in range(1, steps):
            c = ((1,), (2, -1), (3, -3, 1), (4, -6, 4, -1))[len(hist) - 1]
            V, BV = self._step(V, BV, sum(q * v for q, v in zip(c, hist)), ht, theta)
            hist = [V] + hist[:3]
        return V

    def _step(self, V, BV, Y, ht, theta):
        x, q = self.x, ht * theta
        if ht not in self._tables:
            # departure interpolation; each axis' part of the implicit operator inverted on its own
            c0 = math.sqrt(1 + q * self.rw)
            eye = torch.eye(x.size, dtype=torch.float64, device=DEV)
            self._tables[ht] = [_lagrange(x, x * math.exp(k * ht), "linear") for k in self.kappa] + [
                torch.linalg.inv(c0 * eye - 0.5 * q / c0 * s * self.D2) for s in (self.a[0], self.a[2])]
        T1, T2, I1, I2 = self._tables[ht]
        W = T2 @ (V + ht * (1 - theta) * (self.diffuse(V) - self.rw * V + BV)) @ T1.T
        B, last = self.jump(Y), math.inf
        for _ in range(400):
            D = I2 @ (W + q * (B - self.rw * Y + self.diffuse(Y)) - Y) @ I1.T
            Y = Y + D
            size = float(D.abs().max()) / self.K
            B = B + self.jump(D)
            if size < 1e-12 or size >= 0.95 * last and size < 1e-10:
                break
            last = size
        return Y, B


def exact(case, seed):
    kind = case["kind"]
    if kind == "static":
        omega, U = _static_inputs(case, seed)
        n = case["n"]
        s = _LogScheme.__new__(_LogScheme)
        s.n = n
        s._set_weights(omega)
        out = torch.zeros_like(U)
        out[1:n, 1:n] = s.jump(U[1:n, 1:n], 0.0, far=False)
        return out
    if kind in ("jump", "iteration"):
        w, strike = _price_inputs(case, seed)
        n = case["n"]
        s = _LogScheme(_model(w), n, case.get("payoff", 0), strike)
        U = _field(n, seed)
        out = torch.zeros_like(U)
        if kind == "jump":
            out[1:n, 1:n] = s.jump(U[1:n, 1:n], 0.5)
            return out
        delta = torch.zeros_like(U)
        delta[1:n, 1:n] = s.solve_nonmixed((U / 50.0 - 1.0)[1:n, 1:n], 1.0 / 1024, 0.5)
        out[1:n, 1:n] = s.jump(delta[1:n, 1:n], 0.0, far=False)
        return dict(delta=delta, bdelta=out, stop=float((delta.abs() / delta.abs().clamp(min=1.0)).max()))
    if kind == "price":
        w, strike = _price_inputs(case, seed)
        V = _LogScheme(_model(w), case["n"], case["payoff"], strike).solve(case["steps"], case["maturity"],
                                                                          case["sl_order"])
        return dict(price=float(V[case["n"] // 2, case["n"] // 2]), values=V)
    if kind == "batch":
        got = []
        for w, n, steps, K, T in _batch_inputs(case, seed):
            got.append(float(_LogScheme(_model(w), n, 0, K).solve(steps, T)[n // 2, n // 2]))
        return dict(prices=torch.tensor(got, dtype=torch.float64), statuses=None)
    if kind == "adjoint":
        w, strike = _price_inputs(case, seed)
        n = case["n"]

        def price(p):
            v = dict(w, sigma=(p[0], p[1]), corr=p[2], kappa=p[3], beta=(p[4], p[5]))
            return float(_LogScheme(_model(v), n, 0, strike).solve(case["steps"], 1.0)[n // 2, n // 2])

        base = [w["sigma"][0], w["sigma"][1], w["corr"], w["kappa"], w["beta"][0], w["beta"][1]]
        e = 1e-4
        up = [price([v + e * (k == j) for k, v in enumerate(base)]) for j in range(6)]
        dn = [price([v - e * (k == j) for k, v in enumerate(base)]) for j in range(6)]
        grad = torch.tensor([(u - d) / (2 * e) for u, d in zip(up, dn)], dtype=torch.float64)
        return dict(price=torch.tensor(price(base), dtype=torch.float64), grad=grad)
    s = _PriceScheme(case, seed)
    if kind == "space_jump":
        return s.jump(_surface(s.x, s.K, seed))
    return s.solve(case["steps"])
