"""FP64 states out of the fixed-point range: a context whose initial state lies there runs kernels
that update every node in FP64. Its form follows the state, alone, in a batch and from a checkpoint."""
import numpy as np
import pytest

import workloads as wl
from parity_helpers import case_kwargs, check, make_solver

pytestmark = pytest.mark.gpu

N, W = 40, 5


def _kw(q=37, **kw):
    base = dict(nx=N, ny=N, W=W, tau=0.8, sigma_max=0.05, sigma_power=2, bc="nrbc", q=q,
                mean=(1.0, 0.1, 0.05, 1.0))
    base.update(kw)
    return case_kwargs(**base)


def _state(rho0, T0=1.0, W=W):
    r, ux, uy, T = wl.random_smooth_state(N, N, W, seed=3, du=0.02, drho=0.01, dT=0.01,
                                          mean_u=(0.1, 0.05))
    return r * rho0, ux, uy, T + (T0 - 1.0)


INSIDE, OUTSIDE = (1.0, 1.0), (1.0, 1.3)


def _populations(kw, state, calls=(21,)):
    with make_solver(kw, "fp64") as s:
        s.init(*state)
        for n in calls:
            s.step(n)
        return s.export_populations()


@pytest.mark.parametrize("q", [37, 17, 9])
@pytest.mark.parametrize("rho0,T0", [(4.0, 1.0), (0.2, 1.0), (1.0, 1.3)])
@pytest.mark.parametrize("bc,grad,W", [("periodic", "central", 0), ("zg", "central", 5),
                                       ("nrbc", "link", 5)])
def test_outside_everywhere(q, rho0, T0, bc, grad, W):
    kw = _kw(q, bc=bc, pml_grad=grad, W=W, sigma_max=0.05 if W else 0.0,
             mean=(rho0, 0.1, 0.05, T0) if W else (1.0, 0.0, 0.0, 1.0))
    check(kw, _state(rho0, T0, W), 8)


def test_collisionless():
    """omega = 0 keeps populations bit for bit: never in fixed point."""
    kw = _kw(W=0, sigma_max=0.0, bc="periodic", tau=float("inf"), mean=(1.0, 0.0, 0.0, 1.0))
    with make_solver(kw, "fp64") as s:
        s.init(*_state(1.0, W=0))
        M = s.M
        a = s.export_populations()[:, M:M + N, M:M + N]
        s.step(N)                       # every direction is back where it was
        assert np.array_equal(s.export_populations()[:, M:M + N, M:M + N], a)


@pytest.mark.parametrize("first,then", [(INSIDE, OUTSIDE), (OUTSIDE, INSIDE)])
def test_initialized_again_with_another_form(first, then):
    """Graphs of the earlier form are not replayed, alone or in a batch."""
    import torch

    from paper_2504_20169_gb300.serving import Batch

    kw, b = _kw(), _state(*then)
    ref = _populations(kw, b)
    with make_solver(kw, "fp64") as s:
        s.init(*_state(*first))
        s.step(21)
        s.init(*b)
        s.step(21)
        assert np.array_equal(s.export_populations(), ref)
        batch = Batch()
        batch.set([s])
        s.init(*_state(*first))
        batch.step(21)
        torch.cuda.synchronize()
        s.init(*b)
        batch.step(21)
        torch.cuda.synchronize()
        assert np.array_equal(s.export_populations(), ref)
        batch.close()


def test_batch_of_both_forms():
    import torch

    from paper_2504_20169_gb300.serving import Batch

    kw = _kw()
    states = [_state(*INSIDE), _state(*OUTSIDE), _state(1.01), _state(1.0, 1.35)]
    solvers = [make_solver(kw, "fp64") for _ in states]
    try:
        for s, f in zip(solvers, states):
            s.init(*f)
        batch = Batch()
        batch.set(solvers)
        batch.step(21)
        torch.cuda.synchronize()
        batch.close()
        for s, f in zip(solvers, states):
            assert np.array_equal(s.export_populations(), _populations(kw, f))
    finally:
        for s in solvers:
            s.close()


@pytest.mark.parametrize("saved,held", [(INSIDE, OUTSIDE), (OUTSIDE, INSIDE)])
def test_checkpoint_keeps_the_form(saved, held):
    """Restored into a fresh context and into one that ran the other form."""
    kw = _kw()
    with make_solver(kw, "fp64") as s:
        s.init(*_state(*saved))
        s.step(3)
        blob = s.checkpoint()
        s.step(18)
        ref = s.export_populations()
    with make_solver(kw, "fp64") as s:
        s.restore(blob)
        s.step(18)
        assert np.array_equal(s.export_populations(), ref)
        s.init(*_state(*held))
        s.step(18)
        s.restore(blob)
        s.step(18)
        assert np.array_equal(s.export_populations(), ref)
