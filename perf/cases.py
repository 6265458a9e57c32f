"""The work a user of the solver has it do, as measurable cases.

A case is one pass through the public entry points: a whole solve of one problem (from
problem creation to destruction, or on a handle that the program keeps), a batch of
uneven problems, many right-hand sides of one operator, the space-time product on its
own, or a gradient of the learned warm start's network.  Sizes are those of the
repository's configurations, tests and benchmark workloads.

Solutions are computed to the tolerances the tests and the benchmark use (1e-11 below
1023 points in space, 1e-10 from there on, 1e-9 for the precision study), so they
carry many more equal digits than the preconditioner's precision.
"""
from __future__ import annotations

import math
from fractions import Fraction
from types import SimpleNamespace

import numpy as np
import torch

import paper_1305_6653_gb300 as fde

SCHEMES = {"GBDF3": ("GBDF", 3), "GBDF5": ("GBDF", 5), "GAM4": ("GAM", 4), "ETR3": ("ETR", 3)}


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def _solve(name, m, s, alpha, scheme, precision, **more):
    c = {"kind": "solve", "m": m, "s": s, "alpha": alpha, "scheme": scheme, "precision": precision,
         "storage": "fp32", "source": "manufactured", "device": True, "keep": False, "restart": 20,
         "precond": "strang", "timevar": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest calls: the plain FP64 method on 2,016 unknowns (the smoke test's problem),
        # host arrays in and out, one problem from creation to destruction
        _solve("small_fp64", 63, 32, 1.5, "GBDF3", "fp64", device=False),
        # a row of the paper's Tables 1-2 (Example 4.1, n = 96, s = 128), as someone who
        # reproduces the paper runs it
        _solve("paper_fp64", 96, 128, 1.5, "GAM4", "fp64", device=False, source="gaussian"),
        # an ordinary one-off solve on device arrays with the tensor-core preconditioner
        _solve("mid_tf32", 255, 64, 1.7, "GBDF3", "tf32"),
        # the same at a ragged size (m is no multiple of any tile) with FP32 factors
        _solve("ragged_fp32", 700, 128, 1.6, "GBDF5", "fp32"),
        # the benchmark's solve: a kept handle is assembled, factored and solved each time a
        # program's operator changes (TF32 factors, bfloat16 copy for the block solves)
        _solve("scale_tf32", 2047, 256, 1.8, "GBDF5", "tf32", storage="bf16", keep=True, restart=30),
        # the precision study's problem, whose conditioning needs split TF32: the largest factors
        _solve("precision_tf32x3", 4095, 128, 1.9, "GBDF3", "tf32x3", keep=True),
        # the BCCB preconditioner S^(2): no block LU, many cheap iterations
        _solve("bccb_fp64", 1023, 64, 1.5, "GBDF3", "fp64", precond="bccb"),
        # coefficients that vary in time as well
        _solve("timevar_tf32", 511, 128, 1.6, "GBDF5", "tf32", timevar=True),
        # many independent problems of uneven size and scheme in one call
        {"name": "batch_uneven", "kind": "batch", "count": 12, "mix": 0, "precision": "tf32", "storage": "bf16"},
        # many right-hand sides of one operator: one factorisation, grouped block solves
        {"name": "rhs_shared", "kind": "rhs", "m": 1023, "s": 64, "count": 16, "alpha": 1.8, "scheme": "GBDF5",
         "precision": "tf32", "solver": "auto"},
        # the space-time product on its own: a caller with another outer iteration
        {"name": "matvec_fp64", "kind": "matvec", "m": 2047, "s": 256, "alpha": 1.8, "scheme": "GBDF5"},
        # a training step of the learned warm start: forward, loss and every gradient
        {"name": "warmstart_grad", "kind": "grad", "m": 1023, "s": 256, "modes": 16, "width": 64, "layers": 6,
         "ksize": 5, "batch": 32},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "rhs", "matvec", "grad"])
    scheme = rng.choice(["GBDF3", "GBDF5", "GAM4"])
    alpha = round(rng.uniform(1.2, 1.9), 3)
    if kind == "solve":
        precision = rng.choice(["fp64", "fp32", "tf32", "tf32", "tf32x3"])
        precond = "bccb" if precision == "fp64" and rng.random() < 0.3 else "strang"
        s = 1 << rng.randint(4, 8)
        top = {"fp64": 400, "fp32": 1100}.get(precision, 2047)
        m = _log_int(rng, 24, 1100 if precond == "bccb" else top)
        # TF32 updates precondition up to a conditioning h dx^-alpha 2^alpha of about 2e4; the
        # same bound keeps the other solves at the iteration counts of the listed ones
        while 2.0 * (2.0 * (m + 1)) ** alpha / s > 2.0e4:
            m = max(24, int(0.8 * m))
        tc = precision.startswith("tf32")
        return _solve(None, m, s, alpha, scheme, precision, precond=precond,
                      storage=rng.choice(["fp32", "bf16"]) if tc else "fp32",
                      source=rng.choice(["manufactured", "gaussian"]), device=rng.random() < 0.7,
                      keep=rng.random() < 0.5, restart=rng.choice([20, 30]),
                      timevar=precond == "strang" and rng.random() < 0.15)
    if kind == "batch":
        c = {"kind": "batch", "count": rng.randint(4, 12), "mix": rng.randint(1, 10 ** 6),
             "precision": rng.choice(["fp32", "tf32", "tf32"]), "storage": rng.choice(["fp32", "bf16"])}
        while c["count"] > 1 and work(c)["flops"] > (1e12 if c["precision"] == "fp32" else 6e12):
            c["count"] -= 1
        return c
    if kind == "rhs":
        m = _log_int(rng, 100, 1023)
        return {"kind": "rhs", "m": m, "s": 1 << rng.randint(4, 7), "count": rng.randint(3, 16),
                "alpha": round(rng.uniform(1.3, 1.7), 3), "scheme": scheme,
                "precision": rng.choice(["fp32", "tf32"]), "solver": "auto"}
    if kind == "matvec":
        return {"kind": "matvec", "m": _log_int(rng, 24, 4095), "s": 1 << rng.randint(5, 8), "alpha": alpha,
                "scheme": scheme}
    return {"kind": "grad", "m": _log_int(rng, 63, 1023), "s": 1 << rng.randint(4, 8), "modes": rng.choice([8, 16, 32]),
            "width": rng.choice([32, 64]), "layers": rng.randint(3, 6), "ksize": rng.choice([3, 5, 7]),
            "batch": rng.randint(4, 32)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _profile(y, alpha):
    """Riemann-Liouville derivative of y^2 (1-y)^2, lower terminal 0."""
    c = [math.gamma(p + 1) / math.gamma(p + 1 - alpha) for p in (2, 3, 4)]
    return c[0] * y ** (2 - alpha) - 2 * c[1] * y ** (3 - alpha) + c[2] * y ** (4 - alpha)


def _problem(m, s, alpha, scheme, seed, source="manufactured", timevar=False, d=None):
    """One instance of the diffusion problem; the seed varies u0 and the source f.

    manufactured: f of the solution e^-t x^2 (1-x)^2, scaled, plus eight decaying sine modes
    (d+ = 1+x, d- = 2-x).  gaussian: a Gaussian pulse u0 on [0, 2] with f = 0 (d+ = 0.6,
    d- = 0.5).  modes: the sine modes alone, u0 = 0, d+ = d- = d."""
    rng = np.random.default_rng(1305_000 + seed)
    xL, xR, t0, T = 0.0, 2.0 if source == "gaussian" else 1.0, 0.0, 1.0
    x = xL + (xR - xL) / (m + 1) * np.arange(1, m + 1)
    t = np.linspace(t0, T, s + 1)
    dpt = dmt = None
    modes = np.sin(np.pi * np.outer(x, np.arange(1, 9)))
    smooth = np.exp(-rng.uniform(0.5, 2.0) * t)[:, None] * (modes @ rng.standard_normal(8))[None, :]
    if source == "gaussian":
        dp, dm = np.full(m, 0.6), np.full(m, 0.5)
        xc, width = 1.2 + 0.1 * rng.uniform(-1, 1), 0.08 * rng.uniform(0.8, 1.25)
        u0, f = np.exp(-((x - xc) ** 2) / (2 * width ** 2)), np.zeros((s + 1, m))
    elif source == "modes":
        dp, dm = np.full(m, d), np.full(m, d)
        u0, f = np.zeros(m), smooth
    else:
        dp, dm = 1.0 + x, 2.0 - x
        prof = x ** 2 * (1 - x) ** 2
        u0 = prof * (1 + 0.25 * rng.uniform(-1, 1))
        f = (1 + 0.25 * rng.uniform(-1, 1)) * -np.exp(-t)[:, None] * (
            prof + dp * _profile(x, alpha) + dm * _profile(1 - x, alpha))[None, :] + smooth
    if timevar:
        dpt = dp[None, :] * (1 + 0.5 * np.sin(np.pi * t))[:, None]
        dmt = dm[None, :] * (1 + 0.5 * t)[:, None]
        dp, dm = dpt[1:].mean(0), dmt[1:].mean(0)
    family, mu = SCHEMES[scheme]
    p = SimpleNamespace(m=m, s=s, alpha=alpha, xL=xL, xR=xR, t0=t0, T=T, dplus=dp, dminus=dm, u0=u0,
                        f=np.ascontiguousarray(f), family=family, mu=mu)
    if timevar:
        p.dplus_t, p.dminus_t = np.ascontiguousarray(dpt), np.ascontiguousarray(dmt)
    return p


def _solve_problem(case, seed):
    return _problem(case["m"], case["s"], case["alpha"], case["scheme"], seed, case["source"], case["timevar"])


def _tolerance(m):
    return 1e-11 if m < 1023 else 1e-10 if m < 4095 else 1e-9


def _batch_sizes(case):
    """Uneven instances: sizes, orders, schemes and coefficients from the mix."""
    rng = np.random.default_rng(7_000_000 + case["mix"])
    out = []
    for i in range(case["count"]):
        m, s = int(rng.choice((255, 511, 1023, 2047))), int(rng.choice((64, 128, 256)))
        scheme = str(rng.choice(("ETR3", "GBDF3", "GAM4")))
        alpha, d = rng.uniform(1.1, 1.9), rng.uniform(0.5, 2.0)
        # the trapezoidal rule and coarse factors need hundreds of steps on stiff instances
        # (h dx^-alpha large): those keep to a smaller order
        while d * (2.0 * (m + 1)) ** alpha / s > (2.0e3 if scheme == "ETR3" else 2.0e4):
            alpha = 1.0 + 0.9 * (alpha - 1.0)
        out.append((m, s, alpha, scheme, d))
    return out


def _batch_problems(case, seed):
    return [_problem(m, s, alpha, scheme, 64 * seed + i, "modes", d=d)
            for i, (m, s, alpha, scheme, d) in enumerate(_batch_sizes(case))]


def _rhs_problems(case, seed):
    return [_problem(case["m"], case["s"], case["alpha"], case["scheme"], 64 * seed + i) for i in range(case["count"])]


def _network(case, seed):
    """Parameters (He-uniform), inputs and targets of one mini-batch."""
    rng = np.random.default_rng(2_000_000 + seed)
    dims = [case["s"] + 6] + [case["width"]] * (case["layers"] - 1) + [case["s"]]
    theta = []
    for ci, co in zip(dims, dims[1:]):
        b = math.sqrt(6.0 / (ci * case["ksize"]))
        theta += [rng.uniform(-b, b, co * ci * case["ksize"]), 0.01 * rng.standard_normal(co)]
    # sine coefficients fall off with the mode, over the time channels they vary smoothly
    decay = 1.0 / np.arange(1, case["modes"] + 1)
    x = rng.standard_normal((case["batch"], dims[0], case["modes"])) * decay
    y = rng.standard_normal((case["batch"], dims[-1], case["modes"])) * decay
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    return dims, f32(np.concatenate(theta)), f32(x), f32(y)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _fields(p):
    """The problem's arrays and numbers as FDEProblem takes them."""
    f = {k: getattr(p, k) for k in ("m", "s", "alpha", "xL", "xR", "t0", "T", "dplus", "dminus", "u0", "f", "family",
                                    "mu")}
    if hasattr(p, "dplus_t"):
        f.update(dplus_t=p.dplus_t, dminus_t=p.dminus_t)
    return f


def _on_device(f):
    return {k: torch.as_tensor(v, device="cuda") if isinstance(v, np.ndarray) else v for k, v in f.items()}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        f = _fields(_solve_problem(case, seed))
        if case["device"]:
            f = _on_device(f)
        st = SimpleNamespace(case=case, fields=f, handle=None, out=None)
        if case["keep"]:
            st.handle = fde.FDEProblem(**f)
            st.out = torch.empty(case["m"] * case["s"], dtype=torch.float64, device="cuda" if case["device"] else "cpu")
        return st
    if kind == "batch":
        return SimpleNamespace(case=case, problems=_batch_problems(case, seed))
    if kind == "rhs":
        return SimpleNamespace(case=case, problems=_rhs_problems(case, seed))
    if kind == "matvec":
        p = _problem(case["m"], case["s"], case["alpha"], case["scheme"], seed)
        h = fde.FDEProblem(**_on_device(_fields(p))).assemble()
        # a Krylov vector: the right-hand side with a white part
        z = h.rhs()
        g = torch.Generator(device="cuda").manual_seed(seed)
        z = z / z.norm() + torch.randn(z.shape, dtype=z.dtype, device="cuda", generator=g) / math.sqrt(z.numel())
        return SimpleNamespace(case=case, handle=h, z=z)
    _, theta, x, y = _network(case, seed)
    net = fde.FDENop(case["m"], case["s"], modes=case["modes"], width=case["width"], layers=case["layers"],
                     ksize=case["ksize"])
    net.set_params(theta)
    return SimpleNamespace(case=case, net=net, x=torch.from_numpy(x).cuda(), y=torch.from_numpy(y).cuda())


def _assemble_and_solve(p, case, out=None):
    p.assemble()
    if case["precond"] == "bccb":
        p.bccb(precision=case["precision"])
    else:
        p.factor(case["precision"], storage=case["storage"])
    x, _ = p.solve(tol=_tolerance(case["m"]), restart=case["restart"], maxit=2000, out=out)
    return x


def run(st):
    case = st.case
    kind = case["kind"]
    if kind == "solve":
        if st.handle is not None:
            return _assemble_and_solve(st.handle, case, st.out)
        with fde.FDEProblem(**st.fields) as p:
            return _assemble_and_solve(p, case)
    if kind == "batch":
        with fde.FDEBatch(st.problems, device_inputs=True) as b:
            b.assemble().factor(case["precision"], storage=case["storage"])
            xs, _ = b.solve(tol=1e-10, restart=20, maxit=400)
        return xs
    if kind == "rhs":
        with fde.FDEBatch(st.problems, device_inputs=True) as b:
            b.share_operator().block_solver(case["solver"]).assemble().factor(case["precision"])
            xs, _ = b.solve(tol=_tolerance(case["m"]), restart=30, maxit=400)
        return xs
    if kind == "matvec":
        return st.handle.matvec(st.z)
    loss, grad = st.net.loss_grad(st.x, st.y, case["batch"], want_grad=True)
    return {"loss": np.float32(loss), "grad": grad}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _solve_work(m, s, mu, precond="strang", its=10):
    """Bytes: u0, d+-, f in, the solution out.  Flops: the s/2+1 complex LUs, and for `its`
    iterations (the paper's counts, nearly independent of n and s) the block solves, three FFTs of
    length 2m and two of length s with real data, the band, and Gram-Schmidt."""
    n, nk = m * s, s // 2 + 1
    fft = s * 7.5 * 2 * m * math.log2(2 * m) + 5.0 * n * math.log2(s)
    it = fft + 4 * (mu + 1) * n + 4 * its * n
    if precond == "strang":
        it += 8.0 * nk * m * m
    else:
        it += nk * 20.0 * m * math.log2(2 * m)
    lu = 8.0 / 3.0 * nk * m ** 3 if precond == "strang" else 0.0
    return {"bytes": 8.0 * (n + (s + 1) * m + 3 * m), "flops": lu + its * it}


def work(case):
    kind = case["kind"]
    if kind == "solve":
        w = _solve_work(case["m"], case["s"], SCHEMES[case["scheme"]][1], case["precond"])
        if case["timevar"]:
            w["bytes"] += 16.0 * (case["s"] + 1) * case["m"]
        return w
    if kind == "batch":
        ws = [_solve_work(m, s, SCHEMES[scheme][1]) for m, s, _, scheme, _ in _batch_sizes(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "rhs":
        one, lu = _solve_work(case["m"], case["s"], SCHEMES[case["scheme"]][1]), 8.0 / 3.0 * (case["s"] // 2 + 1) * case["m"] ** 3
        return {"bytes": one["bytes"] * case["count"], "flops": lu + case["count"] * (one["flops"] - lu)}
    if kind == "matvec":
        m, s = case["m"], case["s"]
        return {"bytes": 16.0 * m * s, "flops": s * (7.5 * 2 * m * math.log2(2 * m) + 4.0 * (SCHEMES[case["scheme"]][1] + 2) * m)}
    dims = [case["s"] + 6] + [case["width"]] * (case["layers"] - 1) + [case["s"]]
    wts = sum(a * b * case["ksize"] for a, b in zip(dims, dims[1:]))
    # forward, backward to the weights, and backward to the inputs of all but the first layer
    return {"bytes": 4.0 * (2 * wts + case["batch"] * case["modes"] * (dims[0] + dims[-1])),
            "flops": 2.0 * case["batch"] * case["modes"] * (3 * wts - dims[0] * dims[1] * case["ksize"])}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------

def _formula(family, mu, ell):
    """BVM coefficients on the points 0..mu at the point ell from the order conditions."""
    if family == "GBDF":
        beta = [Fraction(int(i == ell)) for i in range(mu + 1)]
        rows = [[Fraction(i) ** q for i in range(mu + 1)] for q in range(mu + 1)]
        rhs = [Fraction(q) * Fraction(ell) ** (q - 1) if q else Fraction(0) for q in range(mu + 1)]
    else:
        alpha = [Fraction(int(i == ell) - int(i == ell - 1)) for i in range(mu + 1)]
        rows = [[q * Fraction(i) ** (q - 1) for i in range(mu + 1)] for q in range(1, mu + 2)]
        rhs = [Fraction(ell) ** q - Fraction(ell - 1) ** q for q in range(1, mu + 2)]
    n = mu + 1
    M = [r + [b] for r, b in zip(rows, rhs)]
    for c in range(n):
        k = next(r for r in range(c, n) if M[r][c] != 0)
        M[c], M[k] = M[k], M[c]
        for r in range(n):
            if r != c and M[r][c] != 0:
                q = M[r][c] / M[c][c]
                M[r] = [x - q * y for x, y in zip(M[r], M[c])]
    sol = [float(M[i][n] / M[i][i]) for i in range(n)]
    return (sol, [float(v) for v in beta]) if family == "GBDF" else ([float(v) for v in alpha], sol)


class _Dense:
    """M of one problem in float64: A (x) I - h B (x) J with dense Toeplitz matrices."""

    def __init__(self, p):
        dev = self.dev = "cuda"
        self.p, m, s, mu = p, p.m, p.s, p.mu
        self.h, dx = (p.T - p.t0) / s, (p.xR - p.xL) / (m + 1)
        nu = mu // 2 + 1 if (p.family == "GBDF" and mu % 2 == 0) else (mu + 1) // 2
        A, B = np.zeros((s + 1, s + 1)), np.zeros((s + 1, s + 1))
        A[0, 0] = 1.0
        cache = {}
        for t in range(1, s + 1):
            at = 0 if t < nu else t - nu if t <= s - mu + nu else s - mu
            a, b = cache.setdefault(t - at, _formula(p.family, mu, t - at))
            A[t, at:at + mu + 1], B[t, at:at + mu + 1] = a, b
        to = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)  # noqa: E731
        self.A, self.B = to(A), to(B)
        g = np.cumprod(np.concatenate([[1.0], 1.0 - (p.alpha + 1.0) / np.arange(1, m + 2)]))
        k = torch.arange(m, device=dev)[:, None] - torch.arange(m, device=dev)[None, :] + 1
        self.G = torch.where(k >= 0, to(g)[k.clamp(min=0)], torch.zeros((), dtype=torch.float64, device=dev)) * dx ** -p.alpha
        self.dp, self.dm = to(p.dplus), to(p.dminus)
        self.t = (to(p.dplus_t), to(p.dminus_t)) if hasattr(p, "dplus_t") else None
        self.J = self.dp[:, None] * self.G + self.dm[:, None] * self.G.T
        a, b = cache[nu] if nu in cache else _formula(p.family, mu, nu)
        w = np.exp(2j * np.pi * np.outer(np.arange(s // 2 + 1), np.arange(mu + 1) - nu) / s)
        self.phi, self.psi = w @ np.array(a), w @ np.array(b)
        u0, f = to(p.u0), to(p.f)
        j0 = self.apply_j(u0[None, :], 0)[0]
        self.b = (self.h * (self.B[1:] @ f) - torch.outer(self.A[1:, 0], u0) + self.h * torch.outer(self.B[1:, 0], j0)).reshape(-1)

    def apply_j(self, z, level):
        """J_n z_n for rows z of the time levels level, level + 1, .."""
        if self.t is None:
            return z @ self.J.T
        n = slice(level, level + z.shape[0])
        return self.t[0][n] * (z @ self.G.T) + self.t[1][n] * (z @ self.G)

    def matvec(self, z):
        z = z.reshape(self.p.s, self.p.m)
        return (self.A[1:, 1:] @ z - self.h * (self.B[1:, 1:] @ self.apply_j(z, 1))).reshape(-1)

    def factor(self):
        m = self.p.m
        kind = torch.complex128 if m <= 300 else torch.complex64  # a preconditioner: its precision is free
        eye, J = torch.eye(m, dtype=kind, device=self.dev), self.J.to(kind)
        self.inv = torch.empty((len(self.phi), m, m), dtype=kind, device=self.dev)
        for k, (a, b) in enumerate(zip(self.phi, self.psi)):
            self.inv[k] = torch.linalg.inv(complex(a) * eye - self.h * complex(b) * J)

    def precond(self, r):
        R = torch.fft.rfft(r.reshape(self.p.s, self.p.m), dim=0)
        Z = torch.bmm(self.inv, R.to(self.inv.dtype)[:, :, None])[:, :, 0]
        return torch.fft.irfft(Z.to(torch.complex128), n=self.p.s, dim=0).reshape(-1)

    def solve(self, cycles=8, steps=24):
        """Flexible GMRES, restarted until the true residual stops falling."""
        self.factor()
        x, best, bx, bn = torch.zeros_like(self.b), math.inf, None, float(self.b.norm())
        for _ in range(cycles):
            r = self.b - self.matvec(x)
            beta = float(r.norm())
            if beta < best:
                better, best, bx = beta < 0.3 * best, beta, x
            else:
                better = False
            if not better or beta <= 1e-14 * bn:
                break
            V, Z, H = [r / beta], [], np.zeros((steps + 1, steps))
            for j in range(steps):
                Z.append(self.precond(V[j]))
                w = self.matvec(Z[j])
                basis = torch.stack(V)
                for _ in range(2):
                    h = basis @ w
                    w = w - h @ basis
                    H[:j + 1, j] += h.cpu().numpy()
                H[j + 1, j] = float(w.norm())
                e = np.zeros(j + 2)
                e[0] = beta
                y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
                if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) <= 1e-5 * beta or H[j + 1, j] == 0:
                    break
                V.append(w / H[j + 1, j])
            x = x + torch.as_tensor(y, device=self.dev) @ torch.stack(Z[:len(y)])
        return bx


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return _Dense(_solve_problem(case, seed)).solve()
    if kind == "batch":
        return [_Dense(p).solve() for p in _batch_problems(case, seed)]
    if kind == "rhs":
        out, first = [], None
        for p in _rhs_problems(case, seed):
            d = _Dense(p)
            if first is None:
                first = d
                d.factor()
            d.factor, d.inv = (lambda: None), first.inv
            out.append(d.solve())
        return out
    if kind == "matvec":
        p = _problem(case["m"], case["s"], case["alpha"], case["scheme"], seed)
        d = _Dense(p)
        z = d.b / d.b.norm()
        g = torch.Generator(device="cuda").manual_seed(seed)
        return d.matvec(z + torch.randn(z.shape, dtype=z.dtype, device="cuda", generator=g) / math.sqrt(z.numel()))
    dims, theta, x, y = _network(case, seed)
    theta = torch.as_tensor(theta, dtype=torch.float64, device="cuda").requires_grad_()
    a, o = torch.as_tensor(x, dtype=torch.float64, device="cuda"), 0
    for i, (ci, co) in enumerate(zip(dims, dims[1:])):
        W = theta[o:o + co * ci * case["ksize"]].reshape(co, ci, case["ksize"])
        o += W.numel()
        a = torch.nn.functional.conv1d(a, W, theta[o:o + co], padding=case["ksize"] // 2)
        o += co
        a = a.relu() if i + 2 < len(dims) else a
    loss = (a - torch.as_tensor(y, dtype=torch.float64, device="cuda")).square().mean()
    return {"loss": loss.detach(), "grad": torch.autograd.grad(loss, theta)[0]}
