"""Digit passes line by line: what a pass makes of a line depends on that line alone, also where several lines are
stacked in one column of a tile (axes of 63 points and fewer).  Whole lines differ by up to 2^1800, a few hold an
infinity or a NaN, and every second one is smooth; each finite line is compared with the plain matrix in extended
precision, on its own scale.

Tolerance, relative to |M||x| of the line: the pass rounds the tabulated operator and the result once each and drops
2^-61 of the line's largest times the operator's largest entry (2^-53 and a little more in all), and the Toeplitz
coefficients and mu are FP64 numbers of some 10 ulp: 2e-15 = 18 2^-53."""
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


def _problem(n):
    d = len(n)
    return W.Problem(d=d, n=n, lo=(-8.0,) * d, hi=(8.0,) * d, alpha=1.5, rho=1.0, dt=0.005)


def _matrices(p, axis):
    """S and mu T_0 of one axis in extended precision."""
    n, N = p.n[axis], p.n[axis] + 1
    j = np.arange(1, n + 1)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    S = np.sqrt(np.longdouble(2) / N) * np.sin(pi * ((j[:, None] * j[None, :]) % (2 * N)).astype(np.longdouble) / N)
    c = [np.longdouble(math.gamma(p.alpha + 1) / math.gamma(p.alpha / 2 + 1) ** 2)]
    for k in range(n - 1):
        c.append(c[-1] * (k - np.longdouble(p.alpha) / 2) / (np.longdouble(p.alpha) / 2 + k + 1))
    mu = np.longdouble(p.dt) / np.longdouble(p.h(axis)) ** np.longdouble(p.alpha)
    return S, mu * np.array(c)[np.abs(j[:, None] - j[None, :])]


def _uneven_lines(p, axis, spread, seed):
    """Base lines (n, lines), a power of two for each line, and the lines that are not finite."""
    rng = np.random.default_rng(seed)
    n = p.n[axis]
    count = p.size // n
    x = rng.standard_normal((n, count)) + 1j * rng.standard_normal((n, count))
    j = np.arange(1, n + 1)[:, None] / (n + 1)
    centre = rng.uniform(0.3, 0.7, count // 2)[None, :]
    x[:, 1::2] = np.exp(-30.0 * (j - centre) ** 2) * (1 + 0.5j)
    e = rng.choice(np.array(spread), count)
    stack = max(1, 128 // (n + 1))
    bad = {1: complex(np.inf, 0.0), 8 * stack + 3: complex(0.0, np.nan), count - 2: complex(1.0, -np.inf)}
    return x, e, bad


def _to_grid(p, axis, lines):
    ax = p.d - 1 - axis
    rest = [m for k, m in enumerate(p.shape) if k != ax]
    return np.ascontiguousarray(np.moveaxis(lines.reshape([p.n[axis]] + rest), 0, ax)).reshape(-1)


def _to_lines(p, axis, grid):
    return np.moveaxis(grid.reshape(p.shape), p.d - 1 - axis, 0).reshape(p.n[axis], -1)


def _check(M, x, e, bad, y, n, tol):
    finite = np.isfinite(y.real) & np.isfinite(y.imag)
    good = np.ones(x.shape[1], dtype=bool)
    good[list(bad)] = False
    assert not finite[:, ~good].any()
    assert finite[:, good].all()
    first = min(x.shape[1], 16 * max(1, 128 // (n + 1)) + 16)  # a whole tile and some of the next
    pick = np.unique(np.concatenate([np.arange(first), np.arange(max(0, x.shape[1] - 48), x.shape[1])]))
    pick = pick[good[pick]]
    xs = x[:, pick]
    want_re, want_im = M @ xs.real.astype(np.longdouble), M @ xs.imag.astype(np.longdouble)
    got_re, got_im = np.ldexp(y[:, pick].real, -e[pick]), np.ldexp(y[:, pick].imag, -e[pick])
    size = np.sqrt(((np.abs(M) @ np.abs(xs).astype(np.longdouble)) ** 2).sum(axis=0))
    err = np.sqrt(((got_re - want_re) ** 2 + (got_im - want_im) ** 2).sum(axis=0)) / size
    assert float(err.max()) < tol, (int(pick[int(err.argmax())]), float(err.max()))


@pytest.mark.parametrize("n", [(3, 127, 255), (7, 255, 63), (63, 15, 127), (127, 3, 255), (255, 7, 63), (31, 63, 31),
                               (511, 127)])
def test_a_line_does_not_depend_on_its_neighbours(n):
    from paper_2410_03643_gb300 import Solver
    p = _problem(n)
    assert p.size >= 60000
    s = Solver(p, precision=0)
    for axis in range(p.d):
        x, e, bad = _uneven_lines(p, axis, [-900, -40, 0, 40, 900], 11 + axis)
        v = np.ldexp(x.real, e) + 1j * np.ldexp(x.imag, e)
        for q, value in bad.items():
            v[n[axis] // 2, q] = value
        v = torch.from_numpy(_to_grid(p, axis, v)).cuda()
        S, T = _matrices(p, axis)
        for M, got in ((S, s.dst(axis, v)), (T, s.toeplitz(axis, v)), (T / 2, s.toeplitz(axis, v, half=True))):
            _check(M, x, e, bad, _to_lines(p, axis, got.cpu().numpy()), n[axis], 2e-15)
    s.close()


@pytest.mark.parametrize("n", [(3, 1023, 511), (7, 511, 511), (15, 511, 255), (255, 3, 2047), (255, 7, 1023), (255, 15, 511),
                               (63, 127, 255), (127, 255, 63)])
def test_fp32_passes_keep_their_lines_apart(n):
    """The same of the FP32 digit passes.  Tolerance: the sum of the leading digits is exact, the two lower ones are
    summed in FP32 2^-11 below it, and the result is rounded once: 4 2^-24 of |M||x|."""
    from paper_2410_03643_gb300 import Solver
    p = _problem(n).replace(restart=2)
    assert p.size >= 1 << 20
    s = Solver(p, precision=1)
    for axis in range(3):
        if n[axis] > 255:
            continue
        x, e, bad = _uneven_lines(p, axis, [-60, -20, 0, 20, 60], 23 + axis)
        x = x.astype(np.complex64)
        v = np.empty(x.shape, dtype=np.complex64)
        v.real, v.imag = np.ldexp(x.real, e), np.ldexp(x.imag, e)
        for q, value in bad.items():
            v[n[axis] // 2, q] = value
        v = torch.from_numpy(_to_grid(p, axis, v)).cuda()
        S, T = _matrices(p, axis)
        x = x.astype(np.complex128)
        for M, op in ((S, 0), (T, 1), (T, 2)):
            y = _to_lines(p, axis, s.test_digit32(axis, op, v).cpu().numpy().astype(np.complex128))
            _check(M, x, e, bad, y, n[axis], 4 * 2.0 ** -24)
    s.close()


def test_mixed_grid_with_an_axis_of_511_points():
    """FP64 residual products as digit passes on an axis whose FP32 passes are FFT passes: two mixed steps against
    the FP64 form, both solved to 1e-10 (1e-8 as everywhere for the mixed form)."""
    from paper_2410_03643_gb300 import Solver
    p = W.Problem(d=3, n=(511, 127, 127), lo=(-6.0,) * 3, hi=(6.0,) * 3, alpha=1.6, rho=1.0, dt=0.01, tol=1e-10, restart=10)
    u0 = torch.from_numpy(W.u0_gaussian(p).reshape(-1).copy()).cuda()
    out = []
    for precision in (1, 0):
        s = Solver(p, precision=precision)
        s.set_state(u0)
        s.run(2)
        out.append(s.get_state()[1])
        s.close()
    assert float((out[0] - out[1]).norm() / out[1].norm()) < 1e-8


def test_fp32_results_keep_their_subnormals_in_fp64():
    """The pass that stores FP64 results stores the FP32 ones, exactly: subnormal, normal and non-finite."""
    from paper_2410_03643_gb300 import Solver
    p = _problem((63, 127, 255)).replace(restart=2)
    s = Solver(p, precision=1)
    for axis in range(3):
        x, e, bad = _uneven_lines(p, axis, [-140, -130, 0], 41 + axis)
        v = np.ldexp(x.real, e) + 1j * np.ldexp(x.imag, e)
        for q, value in bad.items():
            v[0, q] = value
        v = torch.from_numpy(_to_grid(p, axis, v.astype(np.complex64))).cuda()
        single = s.test_digit32(axis, 1, v).cpu().numpy().view(np.float32)
        double = s.test_digit32(axis, 2, v).cpu().numpy().view(np.float64)
        tiny = (single != 0) & (np.abs(single) < np.finfo(np.float32).tiny)
        assert tiny.sum() > p.size // 10
        assert np.array_equal(double, single.astype(np.float64), equal_nan=True)
    s.close()
