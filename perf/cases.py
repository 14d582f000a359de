"""The work that users of this library have it do, as measurable cases.

listed() are the calls of the library's own configurations (forward wavefields, the mixed
256^2 and 512^2 steps, the lower-level FWI evaluation, Hessian products, P2, the autograd
layer, the bilevel hypergradient); draw(rng) gives further sizes of the same ranges.  Every
case goes through the public entry points of paper_2301_10762_gb300 (helm.py, autograd.py).
exact() restates the discrete method in plain 64-bit torch: block elimination line by line
(torch.linalg.inv), one step of iterative refinement, and the method's formulas on top.

Refinement tolerances: 1e-11 for wavefields (a decade under the library's default, so that
they are good to 1e-9 whatever sweep the refinement ends on) and 1e-12 where wavefields go into
gradients (the lower level's own setting).
"""
import math

import numpy as np
import torch

from paper_2301_10762_gb300 import helm as hm
from paper_2301_10762_gb300.autograd import HelmholtzProblem

ALPHA, MU = 1e-3, 1e-6   # regularisation of the hypergradient and of P2 (the FWI-step configuration)
ALPHA_FWI = 1e-6         # of the misfit and Hessian cases (the preconditioner study's smallest): at
                         # 1e-3 the regulariser would drown the data term in the outputs


def listed():
    def case(name, kind, nx, nz, w, nsrc, prec="mixed", rtol=1e-11, nrec=24, **more):
        return {"name": name, "kind": kind, "nx": nx, "nz": nz, "n_omega": w[0], "w_lo": float(w[1]), "w_hi": float(w[2]),
                "nsrc": nsrc, "prec": prec, "rtol": rtol, "nrec": nrec, **more}
    return [
        # one application of the preconditioner P2 = Gamma(alpha0, mu): once per PCG iteration
        case("gamma_128", "gamma", 128, 128, (1, 0, 0), 1, "fp64"),
        # the plain forward problem (64^2, omega = 10, 8 sources) on a resident FP64 factor: the
        # smallest solve, all latency
        case("fp64_solve_64", "solve", 64, 64, (1, 10, 10), 8, "fp64", point=True),
        # assemble + factor + solve with the default precision at the FWI step's size
        case("fp64_step_128", "step", 128, 128, (3, 5, 15), 16, "fp64", point=True),
        # an adjoint solve of dense right-hand sides on a resident mixed factor (the Hessian
        # product's second solve) at the FWI step's size
        case("adjoint_128", "solve", 128, 128, (3, 5, 15), 16, adjoint=True),
        # one right-hand side per frequency on a resident 256^2 factor: a serving call's latency
        case("few_256", "solve", 256, 256, (8, 5, 40), 1, point=True),
        # the headline step: 256^2, 8 frequencies, 64 sources, factor included
        case("step_256", "step", 256, 256, (8, 5, 40), 64, point=True),
        # the same step on 512^2: the largest
        case("step_512", "step", 512, 512, (8, 5, 40), 64, point=True),
        # one phi / grad phi evaluation of the lower level's L-BFGS (new model: assemble, factor,
        # forward and adjoint wavefields, gradient), crosswell, the smallest grid of the uneven set
        case("misfit_96", "misfit", 96, 96, (4, 3, 24), 51, rtol=1e-12),
        # the same on one of its large grids
        case("misfit_224", "misfit", 224, 224, (4, 3, 36), 51, rtol=1e-12),
        # a Hessian product (PCG and preconditioner study) on a middle grid of the uneven set
        case("hessvec_160", "hessvec", 160, 160, (4, 3, 36), 51, rtol=1e-12),
        # forward and backward through the autograd layer on an odd rectangular grid
        case("autograd_150x101", "autograd", 150, 101, (3, 4, 17), 12, rtol=1e-12),
        # one whole hypergradient pass of the FWI-step geometry
        case("hypergrad_128", "hypergrad", 128, 128, (3, 5, 15), 16, rtol=1e-12, nrec=32, n_cg=10),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gamma", "solve", "solve", "step", "step", "misfit", "hessvec", "autograd", "hypergrad"])
    prec = "fp64" if kind == "gamma" or (kind in ("solve", "step") and rng.random() < 0.3) else "mixed"
    hi = {"gamma": 256, "solve": 288 if prec == "mixed" else 160, "step": 400 if prec == "mixed" else 128, "misfit": 256,
          "hessvec": 256, "autograd": 192, "hypergrad": 128}[kind]
    nz = _log_int(rng, 32 if kind != "gamma" else 64, hi)
    nx = min(hi, max(24, int(round(nz * math.exp(rng.uniform(-0.4, 0.4))))))
    if kind in ("misfit", "hessvec", "hypergrad", "step") and rng.random() < 0.5:   # grids of the configurations: square, even
        nz -= nz % 2
        nx = nz
    w_hi = min(40.0, 0.15 * min(nx, nz)) * rng.uniform(0.6, 1.0)
    n_omega = 1 if kind == "gamma" else rng.randint(1, 8 if kind in ("solve", "step") else 4)
    if kind == "hypergrad":
        n_omega, w_hi = 3, min(w_hi, 15.0)
    c = {"kind": kind, "nx": nx, "nz": nz, "n_omega": n_omega, "w_lo": w_hi / 3 if n_omega > 1 else w_hi, "w_hi": w_hi,
         "nsrc": 1 if kind == "gamma" else _log_int(rng, 1 if kind in ("solve", "step") else 8, 64), "prec": prec,
         "rtol": 1e-11 if kind in ("gamma", "solve", "step") else 1e-12, "nrec": rng.randint(16, 32)}
    if kind in ("solve", "step"):
        c["point"] = kind == "step" or rng.random() < 0.5
        c["adjoint"] = kind == "solve" and rng.random() < 0.5
    if kind == "hypergrad":
        c["nsrc"], c["n_cg"] = rng.randint(8, 16), rng.randint(4, 10)
    return c


# ----------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field(nx, nz, lx, gen, corr=0.1):
    """Gaussian random field with correlation length corr on [0, lx] x [0, 1], max |.| = 1 (white
    noise filtered on a padded periodic grid, as in the configurations' velocity models)."""
    hx, hz = lx / (nx - 1), 1.0 / (nz - 1)
    px, pz = nx + math.ceil(4 * corr / hx), nz + math.ceil(4 * corr / hz)
    w = torch.randn(px, pz, generator=gen, device="cuda", dtype=torch.float64)
    kx = 2 * math.pi * torch.fft.fftfreq(px, d=hx, device="cuda", dtype=torch.float64)
    kz = 2 * math.pi * torch.fft.fftfreq(pz, d=hz, device="cuda", dtype=torch.float64)
    amp = torch.exp(-0.25 * corr ** 2 * (kx[:, None] ** 2 + kz[None, :] ** 2))
    g = torch.fft.ifft2(torch.fft.fft2(w) * amp).real[:nx, :nz]
    g = g - g.mean()
    return g / g.abs().max()


def _smoother(n, sigma=4.0):
    """Matrix of a Gaussian smoothing with reflecting ends, sigma in nodes."""
    K = np.zeros((n, n))
    rad = min(int(4 * sigma), n - 1)
    t = np.arange(-rad, rad + 1)
    k = np.exp(-0.5 * (t / sigma) ** 2)
    k /= k.sum()
    for i in range(n):
        j = np.abs(i + t)
        j = np.where(j > n - 1, 2 * (n - 1) - j, j)
        np.add.at(K[i], j, k)
    return torch.tensor(K, device="cuda")


def _inputs(case, seed):
    """Everything a case is given: the model(s), the acquisition, right-hand sides."""
    nx, nz = case["nx"], case["nz"]
    gen, r = _gen(seed), np.random.default_rng(seed)
    lx = (nx - 1) / (nz - 1)
    d = {"lx": lx, "om": np.linspace(case["w_lo"], case["w_hi"], case["n_omega"])}
    n = case["nsrc"]
    if case["kind"] == "gamma":
        d["r"] = torch.randn(nx * nz, generator=gen, device="cuda", dtype=torch.float64)
        return d
    g = _field(nx, nz, lx, gen)
    if case["kind"] in ("autograd", "hypergrad"):   # the FWI step's model: c' = 1 + 0.3 g
        c = 1.0 + 0.3 * g
    else:   # c in [1.5, 4.5], the speeds of the uneven set and of the solve server
        c = 1.5 + 3.0 * (g - g.min()) / (g.max() - g.min())
    if case["kind"] in ("solve", "step"):   # sources on top-row nodes
        d["m"] = (c ** -2).reshape(-1).contiguous()
        i = np.sort(r.integers(1, nx - 1, n))
        d["src"] = np.stack([i * lx / (nx - 1), np.zeros(n)], 1)
        d["rec"] = np.stack([r.uniform(0.05, 0.95, case["nrec"]) * lx, r.uniform(0.05, 0.95, case["nrec"])], 1)
        if not case.get("point"):
            d["B"] = torch.randn(case["n_omega"], n, nx * nz, generator=gen, device="cuda", dtype=torch.complex128)
        return d
    m_true = c ** -2
    d["m_true"] = m_true.reshape(-1).contiguous()
    d["m"] = (_smoother(nx) @ m_true @ _smoother(nz).T).reshape(-1).contiguous()
    if case["kind"] == "hypergrad":   # the FWI step's surface acquisition
        d["src"] = np.stack([np.round((np.arange(n) + 0.5) * (nx - 1) / n) * lx / (nx - 1), np.zeros(n)], 1)
        d["rec"] = np.stack([(np.arange(case["nrec"]) + 0.5 + r.uniform(-0.2, 0.2, case["nrec"])) * lx / case["nrec"],
                             np.zeros(case["nrec"])], 1)
    else:   # crosswell: sources on nodes of a column near x = 0.05, receivers near the far side
        ix = max(1, round(0.05 * (nx - 1)))
        d["src"] = np.stack([np.full(n, ix * lx / (nx - 1)), np.round(np.linspace(0.05, 0.95, n) * (nz - 1)) / (nz - 1)], 1)
        d["rec"] = np.stack([np.full(case["nrec"], 0.95 * lx), r.uniform(0.05, 0.95, case["nrec"])], 1)
    if case["kind"] == "hessvec":
        d["p"] = _field(nx, nz, lx, gen).reshape(-1).contiguous()
    return d


def _prec(case):
    return hm.HELM_FP64 if case["prec"] == "fp64" else hm.HELM_MIXED


def _data(case, d, acq):
    """Receiver data of the true model, from FP64 factors (as the lower-level driver makes them)."""
    op = hm.helm_assemble(case["nx"], case["nz"], d["lx"], 1.0, d["m_true"], d["om"])
    f = hm.helm_factor(op, hm.HELM_FP64)
    U, _ = hm.helm_solve(f, hm.helm_sources(op, acq))
    y = hm.helm_restrict(op, acq, U)
    f.close()
    op.close()
    return y


def prepare(case, seed):
    d = _inputs(case, seed)
    s = {"case": case, "kind": case["kind"], "prec": _prec(case), **d}
    if case["kind"] == "gamma":
        return s
    s["acq"] = acq = hm.Acq(d["src"], d["rec"])
    grid = (case["nx"], case["nz"], d["lx"], 1.0)
    s["grid"] = grid
    if case["kind"] == "solve":
        s["op"] = hm.helm_assemble(*grid, d["m"], d["om"])
        s["f"] = hm.helm_factor(s["op"], s["prec"])
        if case.get("point"):
            s["B"] = hm.helm_sources(s["op"], acq)
    elif case["kind"] in ("misfit", "hessvec", "autograd"):
        s["data"] = _data(case, d, acq)
        if case["kind"] == "hessvec":
            s["op"] = hm.helm_assemble(*grid, d["m"], d["om"])
            s["f"] = hm.helm_factor(s["op"], s["prec"])
            _, _, s["U"], s["Lam"] = hm.fwi_misfit_grad(s["f"], acq, s["data"], ALPHA_FWI, MU, rtol=case["rtol"],
                                                         want_fields=True)
        if case["kind"] == "autograd":
            s["prob"] = HelmholtzProblem(*grid, d["om"], acq=acq, prec=s["prec"], rtol=case["rtol"], max_iter=20)
            s["B"] = s["prob"].sources()
            s["m"] = s["m"].requires_grad_(True)
    return s


def run(s):
    case, kind = s["case"], s["kind"]
    rtol = case["rtol"]
    if kind == "gamma":
        return hm.helm_gamma_solve(case["nx"], case["nz"], ALPHA, MU, s["r"], lx=s["lx"])
    if kind == "solve":
        call = hm.helm_adjoint_solve if case.get("adjoint") else hm.helm_solve
        return call(s["f"], s["B"], rtol=rtol, max_iter=20)[0]
    if kind == "step":
        op = hm.helm_assemble(*s["grid"], s["m"], s["om"])
        f = hm.helm_factor(op, s["prec"])
        X, _ = hm.helm_solve(f, hm.helm_sources(op, s["acq"]), rtol=rtol, max_iter=20)
        f.close()
        op.close()
        return X
    if kind == "misfit":
        op = hm.helm_assemble(*s["grid"], s["m"], s["om"])
        f = hm.helm_factor(op, s["prec"])
        phi, grad, _, _ = hm.fwi_misfit_grad(f, s["acq"], s["data"], ALPHA_FWI, MU, rtol=rtol)
        f.close()
        op.close()
        return {"phi": phi, "grad": grad}
    if kind == "hessvec":
        return hm.fwi_hessian_vec(s["f"], s["acq"], s["U"], s["Lam"], s["p"], ALPHA_FWI, MU, rtol=rtol)
    if kind == "autograd":
        m = s["m"]
        m.grad = None
        y = s["prob"].restrict(s["prob"].solve(m, s["B"]))
        loss = 0.5 * (s["data"] - y).abs().square().sum()
        loss.backward()
        return {"y": y.detach(), "grad_m": m.grad}
    out = hm.bilevel_hypergrad([s["grid"]], [s["m"]], [s["m_true"]], s["acq"], s["om"], ALPHA, ALPHA, MU, s["prec"],
                               cg_fixed_iters=case["n_cg"], refine_rtol=rtol)
    return {k: out[k] for k in ("psi", "dpsi_dalpha", "dpsi_dp", "dpsi_dw")}


# ------------------------------------------------------------------------------- work

def work(case):
    """One pass: the factor read once per triangular half and direction of every solve (what any
    dense line factor needs), the inputs and outputs once; arithmetic of a line-by-line block
    elimination (n_z^3 complex multiply-adds per line) and of one pass of substitutions."""
    nx, nz, nw, ns = case["nx"], case["nz"], case["n_omega"], case["nsrc"]
    N, kind = nx * nz, case["kind"]
    e = 16 if case["prec"] == "fp64" else 8
    if kind == "gamma":
        return {"bytes": 16.0 * N + 8.0 * (nx * nx + nz * nz), "flops": 4.0 * N * (nx + nz)}
    factor_b, solve_b = e * nw * nx * nz ** 2, 32.0 * nw * ns * N
    factor_f, solve_f = 8.0 * nw * nx * nz ** 3, 16.0 * nw * ns * nx * nz ** 2
    factors, solves = {"solve": (0, 1), "step": (1, 1), "misfit": (1, 2), "hessvec": (0, 2), "autograd": (1, 2),
                       "hypergrad": (2, 5 + 2 * case.get("n_cg", 0))}[kind]
    return {"bytes": float(factors * factor_b + solves * (factor_b + solve_b)), "flops": factors * factor_f + solves * solve_f}


# ------------------------------------------------------------- the method in plain 64 bits

class _Exact:
    """A(m, w) for all w by block elimination over lines of constant x, in complex128."""

    def __init__(self, nx, nz, lx, m, om):
        self.nx, self.nz = nx, nz
        f8 = {"dtype": torch.float64, "device": "cuda"}
        hx, hz = lx / (nx - 1), 1.0 / (nz - 1)
        qx, qz = torch.ones(nx, **f8), torch.ones(nz, **f8)
        qx[[0, -1]] = 0.5
        qz[[0, -1]] = 0.5
        ex, ez = (qx == 0.5).double(), (qz == 0.5).double()
        self.m = m.reshape(nx, nz)
        self.om = torch.tensor(om, **f8)[:, None, None]
        self.d = hx * hz * qx[:, None] * qz[None, :]
        self.b = hx * qx[:, None] * ez[None, :] + hz * ex[:, None] * qz[None, :]
        stiff = (hz / hx) * qz[None, :] * (2 - ex)[:, None] + (hx / hz) * qx[:, None] * (2 - ez)[None, :]
        self.diag = torch.complex(stiff - self.om ** 2 * self.d * self.m, -self.om * self.b * self.m.sqrt())
        self.cx, self.cz = -(hz / hx) * qz, -(hx / hz) * qx
        self.g = torch.complex((self.om ** 2 * self.d).expand_as(self.diag.real), self.om * self.b / (2 * self.m.sqrt()))
        self.gp = torch.complex(torch.zeros_like(self.diag.real), -self.om * self.b / (4 * self.m ** 1.5))
        off = torch.diag(torch.ones(nz - 1, **f8), 1)
        off = off + off.T
        G = None
        self.G = torch.empty(len(om), nx, nz, nz, dtype=torch.complex128, device="cuda")
        cc = self.cx[:, None] * self.cx[None, :]
        for i in range(nx):
            S = torch.diag_embed(self.diag[:, i]) + self.cz[i] * off
            if G is not None:
                S = S - cc * G
            G = torch.linalg.inv(S)
            self.G[:, i] = G

    def apply(self, x):
        """A x, x [n_omega, n, nx, nz]."""
        y = self.diag[:, None] * x
        y[:, :, 1:] += self.cx * x[:, :, :-1]
        y[:, :, :-1] += self.cx * x[:, :, 1:]
        y[..., 1:] += self.cz[:, None] * x[..., :-1]
        y[..., :-1] += self.cz[:, None] * x[..., 1:]
        return y

    def _substitute(self, b):
        y = torch.empty_like(b)
        for i in range(self.nx):
            t = b[:, :, i] if i == 0 else b[:, :, i] - self.cx * y[:, :, i - 1]
            y[:, :, i] = t @ self.G[:, i]            # G is complex symmetric
        for i in range(self.nx - 2, -1, -1):
            y[:, :, i] -= (self.cx * y[:, :, i + 1]) @ self.G[:, i]
        return y

    def solve(self, b):
        b = b.reshape(b.shape[0], b.shape[1], self.nx, self.nz)
        x = self._substitute(b)
        x = x + self._substitute(b - self.apply(x))
        return x.reshape(x.shape[0], x.shape[1], -1)

    def adjoint(self, b):
        return self.solve(b.conj().resolve_conj()).conj().resolve_conj()


def _point_sources(case, d):
    nx, nz = case["nx"], case["nz"]
    B = torch.zeros(case["n_omega"], case["nsrc"], nx * nz, dtype=torch.complex128, device="cuda")
    for q, (x, z) in enumerate(d["src"]):
        B[:, q, round(x / d["lx"] * (nx - 1)) * nz + round(z * (nz - 1))] = 1.0
    return B


def _restriction(case, d):
    """The sliding bicubic R and its derivatives in the receiver position, [3][n_rec][N]."""
    nx, nz, lx = case["nx"], case["nz"], d["lx"]

    def axis(t, n):
        i0 = max(0, min(int(math.floor(t)) - 1, n - 4))
        s = t - i0
        w = [math.prod((s - b) / (a - b) for b in range(4) if b != a) for a in range(4)]
        dw = [sum(math.prod(s - b for b in range(4) if b not in (a, c)) for c in range(4) if c != a)
              / math.prod(a - b for b in range(4) if b != a) for a in range(4)]
        return i0, w, dw

    R = np.zeros((3, len(d["rec"]), nx, nz))
    for r, (x, z) in enumerate(d["rec"]):
        hx, hz = lx / (nx - 1), 1.0 / (nz - 1)
        i0, wx, dx = axis(x / hx, nx)
        j0, wz, dz = axis(z / hz, nz)
        R[0, r, i0:i0 + 4, j0:j0 + 4] = np.outer(wx, wz)
        R[1, r, i0:i0 + 4, j0:j0 + 4] = np.outer(dx, wz) / hx
        R[2, r, i0:i0 + 4, j0:j0 + 4] = np.outer(wx, dz) / hz
    return torch.tensor(R.reshape(3, len(d["rec"]), -1), device="cuda").to(torch.complex128)


def _reg(case, v):
    """R v of the regulariser Gamma = alpha R + mu I."""
    nx, nz = case["nx"], case["nz"]
    v = v.reshape(nx, nz)
    out = torch.zeros_like(v)
    dx, dz = (v[1:] - v[:-1]) * (nx - 1) ** 2, (v[:, 1:] - v[:, :-1]) * (nz - 1) ** 2
    out[1:] += dx
    out[:-1] -= dx
    out[:, 1:] += dz
    out[:, :-1] -= dz
    return out.reshape(-1)


def _gamma_inverse(case):
    nx, nz = case["nx"], case["nz"]

    def dct(n):
        a = torch.arange(n, dtype=torch.float64, device="cuda")
        C = torch.cos(math.pi * a[:, None] * (2 * a[None, :] + 1) / (2 * n)) * math.sqrt(2.0 / n)
        C[0] = math.sqrt(1.0 / n)
        return C, (n - 1) ** 2 * (2 - 2 * torch.cos(math.pi * a / n))

    (Cx, lx), (Cz, lz) = dct(nx), dct(nz)

    def once(r):
        T = Cx @ r.reshape(nx, nz) @ Cz.T / (ALPHA * (lx[:, None] + lz[None, :]) + MU)
        return (Cx.T @ T @ Cz).reshape(-1)

    def apply(r):
        z = once(r)
        return z + once(r - ALPHA * _reg(case, z) - MU * z)
    return apply


def exact(case, seed):
    kind = case["kind"]
    d = _inputs(case, seed)
    nx, nz = case["nx"], case["nz"]
    if kind == "gamma":
        return _gamma_inverse(case)(d["r"])
    A = _Exact(nx, nz, d["lx"], d["m"], d["om"])
    B = d["B"] if "B" in d else _point_sources(case, d)
    if kind in ("solve", "step"):
        return A.adjoint(B) if case.get("adjoint") else A.solve(B)
    R, Rx, Rz = _restriction(case, d)
    At = _Exact(nx, nz, d["lx"], d["m_true"], d["om"])
    Ut = At.solve(B)
    del At
    U = A.solve(B)
    eps = (Ut - U) @ R.T
    Lam = A.adjoint(eps @ R)
    g, gp = A.g.reshape(len(d["om"]), 1, -1), A.gp.reshape(len(d["om"]), 1, -1)
    grad = -(g * U * Lam.conj()).real.sum((0, 1))
    if kind == "autograd":
        return {"y": U @ R.T, "grad_m": grad}
    m, alpha = d["m"], ALPHA if kind == "hypergrad" else ALPHA_FWI
    gm = alpha * _reg(case, m) + MU * m
    if kind == "misfit":
        return {"phi": float(0.5 * eps.abs().square().sum() + 0.5 * (m * gm).sum()), "grad": grad + gm}

    def hess(p):
        V = A.solve(g * U * p)
        Z = A.adjoint((V @ R.T) @ R - p * g.conj() * Lam)
        h = (g * U * Z.conj()).real - (g * V * Lam.conj()).real - (gp * U * Lam.conj()).real * p
        return h.sum((0, 1)) + alpha * _reg(case, p) + MU * p

    if kind == "hessvec":
        return hess(d["p"])
    # hypergradient: rho = H^{-1}(m' - m) by preconditioned conjugate gradients from x = 1
    rhs = d["m_true"] - m
    P2 = _gamma_inverse(case)
    x = torch.ones_like(m)
    r = rhs - hess(x)
    z = P2(r)
    p, rz = z, r @ z
    for _ in range(case["n_cg"]):
        h = hess(p)
        a = rz / (p @ h)
        x, r = x + a * p, r - a * h
        z = P2(r)
        rz, old = r @ z, rz
        p = z + rz / old * p
    T = A.solve(g * U * x)
    dU = U - Ut

    def pair(Ra, Rb):
        return ((T @ Ra.T).conj() * (dU @ Rb.T)).real.sum((0, 1))
    return {"psi": float(0.5 * (rhs @ rhs)), "dpsi_dalpha": float(m @ _reg(case, x)),
            "dpsi_dp": torch.stack([pair(Rx, R) + pair(R, Rx), pair(Rz, R) + pair(R, Rz)], 1).cpu().numpy(),
            "dpsi_dw": (2 * pair(R, R)).cpu().numpy()}
