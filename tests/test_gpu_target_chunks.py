"""Characteristic targets of CBC-relax edges, whose tangential terms read the neighbouring chunk's
targets of the old level: the same whether a launch's chunks all run at once or one after another,
and from either of the two target buffers."""
import numpy as np
import pytest

import workloads as wl
from parity_helpers import case_kwargs, make_solver

pytestmark = pytest.mark.gpu

N, STEPS = 400, 9


def _kw(**kw):
    base = dict(nx=N, ny=N, W=0, tau=0.8, sigma_max=0.0, bc="nrbc", nrbc_edges=(1, 1, 1, 1),
                beta=0.2, mean=(1.0, 0.1, 0.05, 1.0))
    base.update(kw)
    return case_kwargs(**base)


def _state(seed, n=N):
    return wl.random_smooth_state(n, n, 0, seed=seed, du=0.02, drho=0.01, dT=0.01,
                                  mean_u=(0.1, 0.05))


@pytest.mark.parametrize("precision", ["fp32dev", "fp64"])
def test_more_chunks_than_fit_at_once(precision):
    """48 members of 52 chunks of 128 threads: 2496 blocks, and 152 SMs hold 16 of them at most."""
    import torch

    from paper_2504_20169_gb300.serving import Batch

    kw, states = _kw(), [_state(k) for k in range(3)]
    alone = []
    for f in states:
        with make_solver(kw, precision) as s:
            s.init(*f)
            s.step(STEPS)
            alone.append(s.export_populations())
    solvers = [make_solver(kw, precision) for _ in range(48)]
    try:
        for m, s in enumerate(solvers):
            s.init(*states[m % 3])
        batch = Batch()
        batch.set(solvers)
        batch.step(STEPS)
        torch.cuda.synchronize()
        batch.close()
        for m, s in enumerate(solvers):
            assert np.array_equal(s.export_populations(), alone[m % 3]), m
    finally:
        for s in solvers:
            s.close()


@pytest.mark.parametrize("precision", ["fp32dev", "fp64"])
@pytest.mark.parametrize("at", [0, 3, 4])
def test_restored_from_either_buffer(precision, at):
    """A checkpoint holds the targets of the current level, whichever buffer they are in."""
    kw, f = _kw(nx=75, ny=75, q=17), _state(5, 75)
    with make_solver(kw, precision) as s:
        s.init(*f)
        s.step(at)
        blob = s.checkpoint()
        s.step(12)
        ref = s.export_populations()
    with make_solver(kw, precision) as s:
        s.restore(blob)
        s.step(5)
        s.step(7)
        assert np.array_equal(s.export_populations(), ref)
