"""How a step is launched does not change what it computes: graphs of eight steps, the steps
before and after them, and the kernels that put four warps to 32 FP64 nodes on small launches."""
import numpy as np
import pytest

import workloads as wl
from parity_helpers import case_kwargs, make_solver

pytestmark = pytest.mark.gpu


def populations(kw, prec, fields, calls):
    with make_solver(kw, prec) as s:
        s.init(*fields)
        for n in calls:
            s.step(n)
        s.sync()
        return s.export_populations()


@pytest.mark.parametrize("prec", ["fp64", "fp32dev"])
@pytest.mark.parametrize("q,bc,grad,W", [(37, "nrbc", "central", 5), (37, "nrbc", "link", 5),
                                         (17, "nrbc", "central", 4), (9, "zg", "link", 3),
                                         (17, "periodic", "central", 0)])
def test_many_steps_equal_single_steps(prec, q, bc, grad, W):
    """step(n) below, at and beyond a graph's length, from both buffer parities, against step(1)."""
    kw = case_kwargs(nx=45, ny=37, W=W, tau=0.8, sigma_max=0.05 if W else 0.0, sigma_power=2, bc=bc,
                     q=q, pml_grad=grad, mean=(1.0, 0.1, 0.05, 1.0))
    f = wl.random_smooth_state(45, 37, W, seed=q, du=0.02, drho=0.01, dT=0.01, mean_u=(0.1, 0.05))
    ref = populations(kw, prec, f, [1] * 30)
    for calls in ([30], [1, 8, 21], [3, 16, 11], [7, 17, 6], [5] * 6):
        assert np.array_equal(populations(kw, prec, f, calls), ref)


@pytest.mark.parametrize("q,grad", [(37, "central"), (17, "link"), (9, "central")])
def test_large_fp64_batch_equals_its_members(q, grad):
    """A batch with more blocks than the split kernels take against members alone, which they do."""
    import torch

    from paper_2504_20169_gb300.serving import Batch

    nx, ny, W, n = 96, 80, 8, 14      # 14 x 24 frame blocks of 128 nodes
    kw = case_kwargs(nx=nx, ny=ny, W=W, tau=0.8, sigma_max=0.05, sigma_power=2, bc="nrbc", q=q,
                     pml_grad=grad, mean=(1.0, 0.1, 0.0, 1.0))
    states = [wl.random_smooth_state(nx, ny, W, seed=m, du=0.02, drho=0.01, dT=0.01,
                                     mean_u=(0.1, 0.0)) for m in range(n)]
    solvers = [make_solver(kw, "fp64") for _ in range(n)]
    try:
        for s, f in zip(solvers, states):
            s.init(*f)
        batch = Batch()
        batch.set(solvers)
        batch.step(11)
        torch.cuda.synchronize()
        batch.close()
        got = [s.export_populations() for s in solvers]
    finally:
        for s in solvers:
            s.close()
    for m in range(n):
        assert np.array_equal(got[m], populations(kw, "fp64", states[m], [11]))


@pytest.mark.parametrize("prec", ["fp64", "fp32dev"])
def test_step_under_capture_is_refused(prec):
    """Refused without spoiling the caller's capture, and the context goes on as if not called."""
    import torch

    from paper_2504_20169_gb300 import Solver
    from paper_2504_20169_gb300._lib import LBMError

    st = torch.cuda.Stream()
    x = torch.zeros(4, device="cuda")
    f = wl.random_smooth_state(30, 26, 4, seed=1, du=0.02, mean_u=(0.1, 0.05))
    args = (30, 26, 4, 0.8, 0.05, 2, "zg", 17, (0, 0, 0, 0), 0.0, (1.0, 0.1, 0.05, 1.0))
    ref, s = (Solver(*args, precision=prec, stream=st) for _ in range(2))
    ref.init(*f)
    ref.step(30)
    s.init(*f)
    s.step(13)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        x += 1
        for n in (1, 17):
            with pytest.raises(LBMError):
                s.step(n)
    g.replay()
    g.replay()
    s.step(17)
    torch.cuda.synchronize()
    assert torch.all(x == 2)
    assert np.array_equal(s.export_populations(), ref.export_populations())
    s.close()
    ref.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32dev"])
def test_repeated_short_calls_equal_single_steps(prec):
    """Calls of 8 to 11 steps: a graph of eight from the second call on, remainders one by one and
    later by graphs of one."""
    kw = case_kwargs(nx=33, ny=29, W=4, tau=0.8, sigma_max=0.05, sigma_power=2, bc="nrbc", q=17,
                     nrbc_edges=(0, 1, 0, 0), beta=0.2, mean=(1.0, 0.1, 0.05, 1.0))
    f = wl.random_smooth_state(33, 29, 4, seed=2, du=0.02, drho=0.01, dT=0.01, mean_u=(0.1, 0.05))
    ref = populations(kw, prec, f, [1] * 99)
    for calls in ([8, 8, 8, 6] * 3 + [9], [9] * 11, [10] * 9 + [9], [11] * 9):
        assert np.array_equal(populations(kw, prec, f, calls), ref)


@pytest.mark.parametrize("q,grad,n", [(37, "central", 26), (17, "link", 26), (9, "central", 70)])
def test_larger_fp64_batch_equals_its_members(q, grad, n):
    """The band too in more blocks than the split kernel takes (above 256; a member has 11, on D2Q9
    4)."""
    import torch

    from paper_2504_20169_gb300.serving import Batch

    kw = case_kwargs(nx=96, ny=80, W=8, tau=0.8, sigma_max=0.05, sigma_power=2, bc="nrbc", q=q,
                     pml_grad=grad, nrbc_edges=(0, 1, 0, 1), beta=0.2, mean=(1.0, 0.1, 0.0, 1.0))
    states = [wl.random_smooth_state(96, 80, 8, seed=m, du=0.02, drho=0.01, dT=0.01,
                                     mean_u=(0.1, 0.0)) for m in range(3)]
    alone = [populations(kw, "fp64", f, [11]) for f in states]
    solvers = [make_solver(kw, "fp64") for _ in range(n)]
    try:
        for m, s in enumerate(solvers):
            s.init(*states[m % 3])
        batch = Batch()
        batch.set(solvers)
        batch.step(11)
        torch.cuda.synchronize()
        batch.close()
        for m, s in enumerate(solvers):
            assert np.array_equal(s.export_populations(), alone[m % 3]), m
    finally:
        for s in solvers:
            s.close()
