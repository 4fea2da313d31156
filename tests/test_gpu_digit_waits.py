"""The bounded waits inside the digit passes give up: reported once, the loops end, the context stays usable.

A wait of each block is told to give up untried, on a healthy GPU: nothing hangs, the pass waits for its own copies and
products in flight and leaves.  The first wait gives up in every block; later ones where a block has as many."""
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
    return W.Problem(d=d, n=n, lo=(-6.0,) * d, hi=(6.0,) * d, alpha=1.6, rho=1.0, dt=0.01, tol=1e-8, restart=10)


def _gives_up(f, must):
    from paper_2410_03643_gb300.rfnse import RFNSE_ETIMEOUT, RfnseError
    try:
        f()
    except RfnseError as e:
        assert e.status == RFNSE_ETIMEOUT
        return
    assert not must


@pytest.mark.parametrize("device_loop", [1, 0])
@pytest.mark.parametrize("n, precision", [((255, 255), 0), ((511, 127), 0), ((127, 31, 63), 0), ((63, 127, 255), 1)])
def test_a_wait_that_gives_up_is_reported_and_the_context_stays_usable(n, precision, device_loop):
    from paper_2410_03643_gb300 import Solver
    from paper_2410_03643_gb300.rfnse import launch_count
    p = _problem(n)
    s = Solver(p, precision=precision, device_loop=device_loop)
    u0 = torch.from_numpy(W.u0_gaussian(p).reshape(-1).copy()).cuda()
    D = (p.rho * p.dt * u0.abs() ** 2).contiguous()

    def everything():
        out = [s.dst(a, u0) for a in range(p.d)] + [s.toeplitz(a, u0) for a in range(p.d)]
        out += [s.apply_A(u0, D), s.apply_prec(u0, D), s.solve(D, u0)[0]]
        s.set_state(u0)
        s.run(2)
        return [o.cpu().numpy() for o in out + [s.get_state()[1]]]

    want = everything()
    for at in (0, 1, 17):
        s.test_give_up(at)
        must = at == 0
        for a in range(p.d):
            _gives_up(lambda: s.dst(a, u0), must)
            _gives_up(lambda: s.toeplitz(a, u0), must)
        if precision == 1:
            z = u0.to(torch.complex64)
            for a in range(p.d):
                for op in range(3):
                    _gives_up(lambda: s.test_digit32(a, op, z), must)
        _gives_up(lambda: s.apply_A(u0, D), must)
        before = launch_count()
        _gives_up(lambda: s.solve(D, u0), must)
        if must:  # one Arnoldi step of at most 20 kernels and a cycle's end, not max_it = 2000 of them
            assert launch_count() - before < 60
        s.set_state(u0)
        _gives_up(lambda: s.run(2), must)
    s.test_give_up(-1)
    for got, ref in zip(everything(), want):
        assert np.array_equal(got, ref)
    s.close()


def test_a_batch_names_the_instance_whose_wait_gave_up():
    from paper_2410_03643_gb300 import Batch
    from paper_2410_03643_gb300.rfnse import RFNSE_ETIMEOUT, RfnseError
    p = _problem((255, 255))
    b = Batch([p, p], precision=0)
    u0 = torch.from_numpy(W.u0_gaussian(p).reshape(-1).copy()).cuda()
    for i in range(2):
        b.set_state(i, u0)
    b.lib.rfnse_test_give_up(b.ctx[1], 0)
    with pytest.raises(RfnseError, match="instance 1") as e:
        b.run(1)
    assert e.value.status == RFNSE_ETIMEOUT
    b.lib.rfnse_test_give_up(b.ctx[1], -1)
    for i in range(2):
        b.set_state(i, u0)
    b.run(3)
    assert torch.equal(b.get_state(0)[1], b.get_state(1)[1])
    b.close()
