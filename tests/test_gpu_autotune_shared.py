"""Tuner choices shared between contexts of one grid: those of a context without digit passes do not decide for one
that has them."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_03643_gb300 import build
    build.build_library()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"


def test_an_fp64_context_keeps_its_digit_passes_after_a_mixed_one_was_tuned():
    """2047 x 255: the mixed form (below 2^20 points) runs its FP64 products as FFT passes, the FP64 form those along y as
    digit passes, three times faster (511^2: 27 against 87 us); the two forms differ in their rounding."""
    from paper_2410_03643_gb300 import Solver
    p = W.Problem(d=2, n=(2047, 255), lo=(-8.0, -8.0), hi=(8.0, 8.0), alpha=1.5, rho=1.0, dt=0.005, restart=5)
    x = torch.from_numpy(W.random_field(p.shape, 5).reshape(-1).copy()).cuda()
    m, f = Solver(p, precision=1), Solver(p, precision=0)
    digits, fft = f.toeplitz(1, x), m.toeplitz(1, x)
    assert not torch.equal(digits, fft)
    m.autotune()
    f.autotune()
    assert torch.equal(m.toeplitz(1, x), fft)
    assert torch.equal(f.toeplitz(1, x), digits)
    m.close()
    f.close()
