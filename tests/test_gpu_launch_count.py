"""rfnse_launch_count of solves that run as graphs: per Arnoldi step as many kernels as the host-driven loop launches
one by one, untuned and with the tuner's choices (which the two contexts of a grid share)."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_03643_gb300 import build
    build.build_library()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"


@pytest.mark.parametrize("n, precision", [((1023,), 1), ((63, 31), 0), ((511, 511), 1), ((511, 511), 0), ((255, 127, 63), 0),
                                          ((127, 255, 63), 1)])
def test_kernels_of_an_arnoldi_step(n, precision):
    from paper_2410_03643_gb300 import NoConvergence, Solver
    from paper_2410_03643_gb300.rfnse import launch_count
    d = len(n)

    def kernels(max_it, device_loop, tuned):
        p = W.Problem(d=d, n=n, lo=(-8.0,) * d, hi=(8.0,) * d, alpha=1.5, rho=1.0, dt=0.005, tol=1e-14, max_it=max_it)
        s = Solver(p, precision=precision, device_loop=device_loop)
        u = torch.from_numpy(W.random_field(p.shape, 3).reshape(-1).copy()).cuda()
        D = (p.rho * p.dt * u.abs() ** 2).contiguous()
        if tuned:
            s.autotune()
        before = launch_count()
        with pytest.raises(NoConvergence):
            s.solve(D, u)
        after = launch_count()
        s.close()
        return after - before

    for tuned in (False, True):
        step = [kernels(3, loop, tuned) - kernels(2, loop, tuned) for loop in (1, 0)]
        assert step[0] == step[1] > 0, tuned
