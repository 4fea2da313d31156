"""The calls that a user of this framework makes, as cases to be timed and compared.

A case is one call pattern ("kind") on one grid:

  run       Solver.set_state(u0), Solver.run(steps), Solver.get_state(): a trajectory from its initial data
  batch     the same for a Batch of independent 2-D instances
  adjoint   Solver.tape_forward and Solver.tape_backward: a run and the gradient of a loss of its end state
  apply_A   Solver.apply_A: the system matrix (D - T + iI) u
  apply_prec  Solver.apply_prec: the sine-transform preconditioner
  dst       Solver.dst: the orthonormal sine transform along one axis
  solve     Solver.solve: one preconditioned GMRES solve with a given diagonal and right-hand side
  tban      Solver.tban_solve: the stationary iteration

precision 0 is the FP64 form, 1 the mixed FP32/FP64 form; n_a + 1 is a power of two on every axis (the
library takes no other grids, so every size is odd), and the axes may differ.  Time stepping runs at the
solver's default tolerance 1e-10 everywhere.  Iteration counts are returned in the FP64 form; in the
mixed form an inner stopping test sees FP32 rounding, so a count is a diagnostic there that may move by
one without the solution changing, and only the states come back.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2410_03643_gb300 as F

DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ---- the cases ----------------------------------------------------------------------------------

def listed():
    return [
        # one line of points, every launch latency: the 1-D soliton run of the 1-D workload, part of its 50 steps
        {"name": "run 1d 1023 mixed", "kind": "run", "nx": 1023, "ny": 1, "nz": 1, "precision": 1, "steps": 20,
         "alpha": 1.5, "rho": 2.0, "dt": 0.01, "half": 20.0},
        # a small anisotropic 2-D grid in FP64: parameter studies, the tests' sizes
        {"name": "run 2d 63x31 fp64", "kind": "run", "nx": 63, "ny": 31, "nz": 1, "precision": 0, "steps": 10,
         "alpha": 1.2, "rho": 2.0, "dt": 0.005, "half": 10.0},
        # the 2-D workload in the mixed form, the grid most runs are done on
        {"name": "run 2d 511 mixed", "kind": "run", "nx": 511, "ny": 511, "nz": 1, "precision": 1, "steps": 10,
         "alpha": 1.5, "rho": 2.0, "dt": 0.005, "half": 10.0},
        # the same grid in FP64 with the hardest of the workload's exponents
        {"name": "run 2d 511 fp64", "kind": "run", "nx": 511, "ny": 511, "nz": 1, "precision": 0, "steps": 4,
         "alpha": 1.9, "rho": 2.0, "dt": 0.005, "half": 10.0},
        # the 3-D workload in the mixed form: the largest grid that is run in earnest
        {"name": "run 3d 255 mixed", "kind": "run", "nx": 255, "ny": 255, "nz": 255, "precision": 1, "steps": 3,
         "alpha": 1.7, "rho": 1.0, "dt": 0.01, "half": 8.0},
        # a ragged 3-D grid in FP64
        {"name": "run 3d 127x255x63 fp64", "kind": "run", "nx": 127, "ny": 255, "nz": 63, "precision": 0, "steps": 3,
         "alpha": 1.7, "rho": 1.0, "dt": 0.01, "half": 8.0},
        # a parameter sweep: uneven 2-D instances advanced together (the batched workload, a quarter of its count)
        {"name": "batch 16 mixed", "kind": "batch", "count": 16, "precision": 1, "steps": 5, "pick": 2410},
        # the gradient workload: 20 steps forward with the tape, then the reverse pass
        {"name": "adjoint 2d 255 fp64", "kind": "adjoint", "nx": 255, "ny": 255, "nz": 1, "precision": 0, "steps": 20,
         "alpha": 1.5, "rho": 2.0, "dt": 0.005, "half": 10.0},
        # one application of the system matrix, for callers with their own outer method: 3-D, FP64
        {"name": "apply_A 3d 255", "kind": "apply_A", "nx": 255, "ny": 255, "nz": 255, "precision": 0,
         "alpha": 1.7, "rho": 1.0, "dt": 0.01, "half": 8.0},
        # one application of the preconditioner, 2-D, FP64
        {"name": "apply_prec 2d 511", "kind": "apply_prec", "nx": 511, "ny": 511, "nz": 1, "precision": 0,
         "alpha": 1.5, "rho": 2.0, "dt": 0.005, "half": 10.0},
        # one mixed solve with a given diagonal and right-hand side on an oblong grid
        {"name": "solve 2d 255x1023 mixed", "kind": "solve", "nx": 255, "ny": 1023, "nz": 1, "precision": 1,
         "alpha": 1.5, "rho": 2.0, "dt": 0.005, "half": 10.0},
        # the paper's stationary iteration, FP64
        {"name": "tban 2d 255x127 fp64", "kind": "tban", "nx": 255, "ny": 127, "nz": 1, "precision": 0,
         "alpha": 1.5, "rho": 2.0, "dt": 0.005, "half": 10.0},
    ]


def draw(rng):
    """One more case: grids whose exponents are spread evenly over the range, every kind and both precisions."""
    kind = rng.choice(["run", "run", "run", "batch", "adjoint", "apply_A", "apply_prec", "dst", "solve", "tban"])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 16), "precision": rng.choice([1, 1, 0]), "steps": rng.randint(2, 5),
                "pick": rng.randrange(1, 1 << 30)}
    precision = rng.choice([0, 1])
    if kind in ("apply_A", "apply_prec", "dst", "tban"):
        precision = 0
    d = rng.choice([1, 2, 2, 3])
    steps = rng.randint(2, 12)
    if d == 1:
        n = [(1 << rng.randint(5, 11)) - 1, 1, 1]
    elif d == 2:
        n = [(1 << rng.randint(4, 10)) - 1, (1 << rng.randint(4, 10)) - 1, 1]
    else:
        n = [(1 << rng.randint(3, 8)) - 1 for _ in range(3)]
        steps = rng.randint(2, 3)
    most = 1 << (21 if kind in ("run", "solve", "tban", "adjoint") and precision == 0 else 24)
    if kind == "adjoint":
        most = 1 << 18
    while n[0] * n[1] * n[2] > most:  # the long FP64 and reverse passes stay below the largest listed case
        a = n.index(max(n))
        n[a] = (n[a] - 1) // 2
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "precision": precision,
         "alpha": round(rng.uniform(1.1, 1.95), 3), "rho": round(rng.uniform(0.5, 3.0), 3),
         "dt": 0.01 if d != 2 else 0.005, "half": {1: 20.0, 2: 10.0, 3: 8.0}[d]}
    if kind in ("run", "adjoint"):
        c["steps"] = steps
    if kind == "dst":
        c["axis"] = rng.randrange(d)
    return c


# ---- problems and inputs ------------------------------------------------------------------------

def _problem(nx, ny, nz, alpha, rho, dt, half):
    n = tuple(v for v in (nx, ny, nz) if v > 1)
    d = len(n)
    return SimpleNamespace(d=d, n=n, lo=(-half,) * d, hi=(half,) * d, alpha=alpha, rho=rho, dt=dt, omega=1.0, restart=20,
                           max_it=2000, tol=1e-10, first_step=1, precond=0, size=nx * ny * nz)


def _of(case):
    return _problem(*(case[k] for k in ("nx", "ny", "nz", "alpha", "rho", "dt", "half")))


def _instances(case):
    """The batch's problems, as a sweep over grids and model parameters draws them."""
    r = np.random.default_rng(case["pick"])
    ps = []
    for _ in range(case["count"]):
        nx, ny = (int(v) for v in r.choice([127, 255, 511], size=2))
        ps.append(_problem(nx, ny, 1, float(r.uniform(1.1, 1.95)), float(r.uniform(0.5, 3.0)), 0.005, 10.0))
    return ps


def _u0(p, rng):
    """A localised wave packet, flat, x fastest: prod sech(x_a - c_a) in 1-D and 2-D, a Gaussian in 3-D, each with a
    plane-wave phase; centres and slopes from the seed."""
    u = torch.ones(1, dtype=torch.complex128, device=DEV)
    for a in range(p.d):  # x first: each further axis is slower
        h = (p.hi[a] - p.lo[a]) / (p.n[a] + 1)
        x = p.lo[a] + h * torch.arange(1, p.n[a] + 1, dtype=torch.float64, device=DEV)
        c, k = float(rng.uniform(-1, 1)), float(rng.uniform(-3, 3) if p.d < 3 else rng.uniform(-1, 1))
        amp = 1 / torch.cosh(x - c) if p.d < 3 else torch.exp(-0.5 * (x - c) ** 2)
        u = (torch.polar(amp, k * x)[:, None] * u[None, :]).reshape(-1)
    return u


def _noisy(u, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    xi = torch.randn(u.numel(), 2, dtype=torch.float64, device=DEV, generator=g)
    return u * (1 + 0.01 * torch.view_as_complex(xi))


def _inputs(case, seed):
    """What the call is given, by name."""
    rng = np.random.default_rng([seed, 77])
    if case["kind"] == "batch":
        return {"u0": [_u0(p, rng) for p in _instances(case)]}
    p = _of(case)
    u = _u0(p, rng)
    if case["kind"] == "run":
        return {"u0": u}
    if case["kind"] == "adjoint":  # the loss |u^N - target|^2 is taken against a nearby wave packet
        return {"u0": u, "g": 2 * (u - _noisy(u, seed))}
    return {"D": p.rho * p.dt * (u.real ** 2 + u.imag ** 2), "v": _noisy(u, seed + 1)}


def prepare(case, seed):
    i = _inputs(case, seed)
    if case["kind"] == "batch":
        h = F.Batch(_instances(case), precision=case["precision"])
    else:
        h = F.Solver(_of(case), precision=case["precision"])
    return {"case": case, "h": h, **i}


def run(state):
    case, h = state["case"], state["h"]
    kind, fp64 = case["kind"], case["precision"] == 0
    if kind == "run":
        h.set_state(state["u0"])
        iters, _ = h.run(case["steps"])
        prev, cur, _ = h.get_state()
        return [prev, cur] + ([iters] if fp64 else [])
    if kind == "batch":
        for i, u in enumerate(state["u0"]):
            h.set_state(i, u)
        iters, _ = h.run(case["steps"])
        return [list(h.get_state(i)[:2]) for i in range(h.count)] + ([iters] if fp64 else [])
    if kind == "adjoint":
        end, iters = h.tape_forward(state["u0"], case["steps"], 5)
        g0, grho, _ = h.tape_backward(state["g"])
        return [end, g0, grho] + ([iters] if fp64 else [])
    if kind == "apply_A":
        return h.apply_A(state["v"], state["D"])
    if kind == "apply_prec":
        return h.apply_prec(state["v"], state["D"])
    if kind == "dst":
        return h.dst(case["axis"], state["v"])
    u, it, _ = (h.solve if kind == "solve" else h.tban_solve)(state["D"], state["v"])
    return [u] + ([it] if fp64 else [])


# ---- the work that cannot be left out -----------------------------------------------------------

def _fft_flops(p):
    """Flops of one complex FFT of length 2(n + 1) for every line of each axis."""
    return sum(p.size / n * 5.0 * 2 * (n + 1) * math.log2(2 * (n + 1)) for n in p.n)


def work(case):
    """Inputs once, outputs once; flops of the transforms, by the FFT, of the few iterations that a solve needs."""
    ps = _instances(case) if case["kind"] == "batch" else [_of(case)]
    its, per_it = 5, 4.0  # a solve; per Arnoldi step two sine transforms and one Toeplitz product (two FFTs)
    b = f = 0.0
    for p in ps:
        if case["kind"] in ("run", "batch"):  # u^{n-1} and u^n in, u^{n+1} out in each step
            b += 48.0 * p.size * case["steps"]
            f += _fft_flops(p) * per_it * its * (case["steps"] + 1)
        elif case["kind"] == "adjoint":
            b += 2 * 48.0 * p.size * case["steps"]
            f += _fft_flops(p) * per_it * its * 2 * (case["steps"] + 1)
        elif case["kind"] == "dst":
            b += 32.0 * p.size
            f += p.size / p.n[case["axis"]] * 10.0 * (p.n[case["axis"]] + 1) * math.log2(2 * (p.n[case["axis"]] + 1))
        else:  # a vector and the diagonal in, a vector out
            b += 40.0 * p.size
            f += _fft_flops(p) * (2.0 if case["kind"] in ("apply_A", "apply_prec") else per_it * its)
    return {"bytes": b, "flops": f}


# ---- the same in plain torch, 64 bits -----------------------------------------------------------

class _Dense:
    """T, S and the scheme of one problem with dense matrices per axis; vectors are flat, x fastest."""

    def __init__(self, p):
        self.p = p
        self.shape = tuple(reversed(p.n))
        self.T, self.S, lam = [], [], torch.zeros(self.shape, dtype=torch.float64, device=DEV)
        for a, n in enumerate(p.n):
            c = [math.gamma(p.alpha + 1) / math.gamma(p.alpha / 2 + 1) ** 2]
            for k in range(n - 1):
                c.append(c[-1] * (k - p.alpha / 2) / (p.alpha / 2 + k + 1))
            c = torch.tensor(c, dtype=torch.float64, device=DEV)
            i = torch.arange(n, device=DEV)
            mu = p.dt / ((p.hi[a] - p.lo[a]) / (n + 1)) ** p.alpha
            self.T.append(mu * c[(i[:, None] - i[None, :]).abs()])
            k = i + 1
            ang = math.pi / (n + 1)
            self.S.append(math.sqrt(2 / (n + 1)) * torch.sin(ang * ((k[:, None] * k[None, :]) % (2 * (n + 1))).double()))
            cosines = torch.cos(ang * ((k[:, None] * i[None, 1:]) % (2 * (n + 1))).double())
            lam = lam + (mu * (c[0] + 2 * cosines @ c[1:])).reshape([-1 if b == a else 1 for b in range(p.d - 1, -1, -1)])
        self.lam = lam

    def along(self, a, M, v):
        """M times every line of axis a (0 is x)."""
        w = torch.view_as_real(v.reshape(self.shape)).movedim(self.p.d - 1 - a, 0)
        return torch.view_as_complex((M @ w.reshape(w.shape[0], -1)).reshape(w.shape).movedim(0, self.p.d - 1 - a).contiguous()).reshape(-1)

    def mulT(self, v):
        return sum(self.along(a, T, v) for a, T in enumerate(self.T))

    def A(self, v, D, s):
        """(D - s T + iI) v"""
        return (D + 1j) * v - s * self.mulT(v)

    def sines(self, v):
        for a, S in enumerate(self.S):
            v = self.along(a, S, v)
        return v

    def prec(self, v, D, s):
        """2w ((w + 1) - iD)^-1 S (w + i s Lambda)^-1 S v"""
        w = self.p.omega
        y = self.sines(self.sines(v) / (w + 1j * s * self.lam.reshape(-1)))
        return 2 * w * y / (w + 1 - 1j * D)

    def solve(self, D, b, s=1.0, tol=1e-13):
        """(D - sT + iI)^-1 b: right-preconditioned GMRES on I + i(sT - D), restarted on the true residual."""
        f = -1j * b
        R = lambda v: -1j * self.A(v, D, s)  # noqa: E731
        x, norm = torch.zeros_like(f), f.norm()
        if norm == 0:
            return x
        for _ in range(4):
            r = f - R(x)
            beta = r.norm()
            if beta < tol * norm:
                break
            V, Z, H = [r / beta], [], np.zeros((31, 30), dtype=complex)
            for j in range(30):
                Z.append(self.prec(V[j], D, s))
                w = R(Z[j])
                for _ in range(2):
                    for i in range(j + 1):
                        h = torch.vdot(V[i], w)
                        H[i, j] += complex(h)
                        w = w - h * V[i]
                H[j + 1, j] = float(w.norm())
                e = np.zeros(j + 2, dtype=complex)
                e[0] = float(beta)
                y, left = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[:2]
                off = np.linalg.norm(H[:j + 2, :j + 1] @ y - e)
                if off < 0.1 * tol * float(norm) or H[j + 1, j].real < 1e-300:
                    break
                V.append(w / H[j + 1, j].real)
            for z, c in zip(Z, y):
                x = x + complex(c) * z
        return x

    def first(self, u0):
        """The Crank-Nicolson first step: (predictor, u^1), with the diagonals of both."""
        k = 0.5 * self.p.rho * self.p.dt
        sols = []
        at = u0
        for _ in range(2):
            D = k * (at.real ** 2 + at.imag ** 2)
            u = self.solve(D, -self.A(u0, D, 0.5) + 2j * u0, 0.5)
            sols.append((u, D))
            at = (u0 + u) / 2
        return sols

    def forward(self, u0, steps):
        us = [u0]
        for n in range(steps):
            if n == 0:
                us.append(self.first(u0)[1][0])
            else:
                D = self.p.rho * self.p.dt * (us[-1].real ** 2 + us[-1].imag ** 2)
                us.append(self.solve(D, -self.A(us[-2], D, 1.0) + 2j * us[-2]))
        return us

    def back(self, us, g):
        """(dL/du^0, dL/drho) from g = dL/du^N, by the transposed steps."""
        p, N = self.p, len(us) - 1
        grho, grads = 0.0, [torch.zeros_like(g) for _ in us]
        grads[N] = g

        def step(D, s, new, old, gnew):
            """(N^H lam, dL/dD) of M new = N old, M = D - sT + iI, N = -M + 2iI, lam = M^-H gnew."""
            lam = self.solve(D, gnew.conj(), s).conj()  # M is complex symmetric
            dD = -(lam.conj() * (new + old)).real
            return -self.A(lam.conj(), D, s).conj() - 2j * lam, dD

        for n in range(N - 1, 0, -1):
            a2 = us[n].real ** 2 + us[n].imag ** 2
            back, dD = step(p.rho * p.dt * a2, 1.0, us[n + 1], us[n - 1], grads[n + 1])
            grads[n - 1] = grads[n - 1] + back
            grads[n] = grads[n] + 2 * p.rho * p.dt * dD * us[n]
            grho += p.dt * float((dD * a2).sum())
        (u1p, D1), (u1, D2) = self.first(us[0])
        mid = (us[0] + u1p) / 2
        back, dD = step(D2, 0.5, u1, us[0], grads[1])
        g0 = grads[0] + back
        k = 0.5 * p.dt
        grho += k * float((dD * (mid.real ** 2 + mid.imag ** 2)).sum())
        gmid = 2 * p.rho * k * dD * mid
        g0 = g0 + gmid / 2
        back, dD = step(D1, 0.5, u1p, us[0], gmid / 2)
        grho += k * float((dD * (us[0].real ** 2 + us[0].imag ** 2)).sum())
        return g0 + back + 2 * p.rho * k * dD * us[0], grho


def exact(case, seed):
    i = _inputs(case, seed)
    if case["kind"] == "batch":
        ends = [_Dense(p).forward(u, case["steps"])[-2:] for p, u in zip(_instances(case), i["u0"])]
        return ends + ([None] if case["precision"] == 0 else [])
    m = _Dense(_of(case))
    more = [None] if case["precision"] == 0 else []
    if case["kind"] == "run":
        return m.forward(i["u0"], case["steps"])[-2:] + more
    if case["kind"] == "adjoint":
        us = m.forward(i["u0"], case["steps"])
        return [us[-1], *m.back(us, i["g"])] + more
    if case["kind"] == "apply_A":
        return m.A(i["v"], i["D"], 1.0)
    if case["kind"] == "apply_prec":
        return m.prec(i["v"], i["D"], 1.0)
    if case["kind"] == "dst":
        return m.along(case["axis"], m.S[case["axis"]], i["v"])
    return [m.solve(i["D"], i["v"])] + more
