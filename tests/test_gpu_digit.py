"""Digit passes (tensor-core products of FP16 digits) of the FP64 form: S and T along every axis against
the plain matrices in extended precision, at the edges of their tiles: stacked short lines, the unfolded
127, the folded 255 and 511, ragged last tiles on contiguous and strided axes.

Tolerance: the pass rounds the tabulated operator and the result once each (2^-53 relative to entries and
result) and drops 2^-61 of the line's largest times the operator's largest entry; 2e-15 is over ten times
that for random lines (for T also the FP64 rounding of the coefficients themselves, some 10 ulp)."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_03643_gb300 import build
    build.build_library()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"


def _matrices(p, axis):
    n, N = p.n[axis], p.n[axis] + 1
    j = np.arange(1, n + 1)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    S = np.sqrt(np.longdouble(2) / N) * np.sin(pi * ((j[:, None] * j[None, :]) % (2 * N)).astype(np.longdouble) / N)
    c = [np.longdouble(math.gamma(p.alpha + 1) / math.gamma(p.alpha / 2 + 1) ** 2)]
    for k in range(n - 1):
        c.append(c[-1] * (k - np.longdouble(p.alpha) / 2) / (np.longdouble(p.alpha) / 2 + k + 1))
    mu = np.longdouble(p.dt) / np.longdouble(p.h(axis)) ** np.longdouble(p.alpha)
    return S, mu * np.array(c)[np.abs(j[:, None] - j[None, :])]


@pytest.mark.parametrize("n", [(255, 255), (511, 127), (127, 511), (3, 127, 255), (7, 255, 63), (63, 15, 127), (31, 63, 31)])
def test_digit_passes_match_the_matrices(n):
    from paper_2410_03643_gb300 import Solver
    d = len(n)
    p = W.Problem(d=d, n=n, lo=(-8.0,) * d, hi=(8.0,) * d, alpha=1.5, rho=1.0, dt=0.005)
    assert p.size >= 60000
    s = Solver(p, precision=0)
    x = W.random_field(p.shape, 7)
    x.reshape(-1)[:: 97] *= 1e6                      # lines of very uneven magnitude
    v = torch.from_numpy(x.reshape(-1).copy()).cuda()
    for axis in range(d):
        ax = d - 1 - axis
        lines = np.moveaxis(x, ax, 0).reshape(n[axis], -1)
        pick = np.unique(np.concatenate([np.arange(0, lines.shape[1], max(1, lines.shape[1] // 40)),
                                         [lines.shape[1] - 1]]))
        S, T = _matrices(p, axis)
        for M, half, got in ((S, 1, s.dst(axis, v)), (T, 1, s.toeplitz(axis, v)), (T, 2, s.toeplitz(axis, v, half=True))):
            y = np.moveaxis(got.cpu().numpy().reshape(p.shape), ax, 0).reshape(n[axis], -1)[:, pick]
            e_re, e_im = M @ lines[:, pick].real / half, M @ lines[:, pick].imag / half
            err = np.sqrt(float(((y.real - e_re) ** 2 + (y.imag - e_im) ** 2).sum() / (e_re ** 2 + e_im ** 2).sum()))
            assert err < 2e-15, (axis, half, err)
    s.close()


def test_digit_passes_at_the_ends_of_the_number_range():
    """A zero line, subnormal and huge lines, and one line with an infinity: only that line is NaN."""
    from paper_2410_03643_gb300 import Solver
    p = W.Problem(d=2, n=(255, 255), lo=(-8.0, -8.0), hi=(8.0, 8.0), alpha=1.5, rho=1.0, dt=0.005)
    s = Solver(p, precision=0)
    x = W.random_field(p.shape, 9)
    x[0] = 0
    x[1] *= 1e-310
    x[2] *= 1e300
    x[3, 17] = complex(np.inf, 0.0)
    x[4, 0] = complex(0.0, np.nan)
    y = s.dst(0, torch.from_numpy(x.reshape(-1).copy()).cuda()).cpu().numpy().reshape(p.shape)
    S, _ = _matrices(p, 0)
    ok = [r for r in range(255) if r not in (3, 4)]
    assert np.all(y[0] == 0)
    assert not np.any(np.isfinite(y[3].real)) and not np.any(np.isfinite(y[4].imag))
    for r in ok[2:]:
        e = x[r].real @ S
        assert np.linalg.norm((y[r].real - e).astype(float) / 1e300) <= 2e-15 * np.linalg.norm((e / 1e300).astype(float))
    # subnormal results are truncated to a multiple of 2^-1074, and their inputs are
    assert np.max(np.abs(y[1].real - (x[1].real.astype(np.longdouble) @ S).astype(float))) < 20 * 5e-324
    s.close()


@pytest.mark.parametrize("n", [(255, 63, 127), (127, 255, 63), (31, 255, 255)])
def test_fp32_digit_passes_in_the_mixed_form(n):
    """Grids of 2^20 points and more: the FP32 preconditioner against the FP64 one (three FP32 roundings per
    pass, 7 passes: 1e-6 is five times their sum), and two mixed steps against the FP64 form (both solved to
    1e-10, so 1e-8 as everywhere for the mixed form)."""
    from paper_2410_03643_gb300 import Solver
    p = W.Problem(d=3, n=n, lo=(-6.0,) * 3, hi=(6.0,) * 3, alpha=1.6, rho=1.0, dt=0.01, tol=1e-10)
    assert p.size >= 1 << 20
    u0 = torch.from_numpy(W.u0_gaussian(p).reshape(-1).copy()).cuda()
    m, f = Solver(p, precision=1), Solver(p, precision=0)
    D = (p.rho * p.dt * u0.abs() ** 2).contiguous()
    v = torch.from_numpy(W.random_field(p.shape, 5).reshape(-1).copy()).cuda()
    a, b = m.apply_prec(v, D, precision=1), f.apply_prec(v, D)
    assert float((a - b).norm() / b.norm()) < 1e-6
    out = []
    for s in (m, f):
        s.set_state(u0)
        its, _ = s.run(2)
        out.append((s.get_state()[1], its))
        s.close()
    assert float((out[0][0] - out[1][0]).norm() / out[1][0].norm()) < 1e-8
    assert np.all(np.abs(out[0][1].astype(int) - out[1][1].astype(int)) <= 4)
