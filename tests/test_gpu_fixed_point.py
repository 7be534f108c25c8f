"""FP64 grids at the edges of the fixed-point node update: states just inside and outside its
range, densities far from one, negative populations, and every kernel that uses it."""
import numpy as np
import pytest

import workloads as wl
from parity_helpers import case_kwargs, check, make_solver

pytestmark = pytest.mark.gpu

SIZES = dict(nx=37, ny=33, W=5)


def fields(seed, rho0, u0, T0, du=0.03, drho=0.01, dT=0.01, W=5):
    r, ux, uy, T = wl.random_smooth_state(37, 33, W, seed=seed, du=du, drho=drho, dT=dT,
                                          mean_u=u0)
    return r * rho0, ux, uy, T + (T0 - 1.0)


@pytest.mark.parametrize("q", [37, 17, 9])
@pytest.mark.parametrize("rho0,u0,T0", [
    (1.0, (0.45, 0.1), 1.0),       # fast: the outer shells near and below zero on D2Q17 and D2Q9
    (1.0, (0.1, 0.05), 1.235),     # across the upper temperature bound
    (1.0, (0.1, 0.05), 0.765),     # across the lower one
    (3.7, (0.1, 0.0), 1.0),        # another density exponent
    (1.95, (0.05, 0.0), 1.0),      # mean 1, density near the upper bound of its exponent
    (0.51, (0.05, 0.0), 1.0)])     # and near the lower one
@pytest.mark.parametrize("bc,grad", [("zg", "central"), ("nrbc", "link")])
def test_edges_of_the_range(q, rho0, u0, T0, bc, grad):
    """Nodes on both sides of the range in one grid (fixed point inside, FP64 outside)."""
    mean_rho = rho0 if rho0 > 2 else 1.0
    kw = case_kwargs(tau=0.8, sigma_max=0.05, sigma_power=2, bc=bc, q=q, pml_grad=grad,
                     mean=(mean_rho, u0[0], u0[1], T0), **SIZES)
    check(kw, fields(q, rho0, u0, T0), 6)


@pytest.mark.parametrize("q", [37, 17])
def test_negative_and_small_populations(q):
    """Populations that are negative, zero or far below their weight."""
    kw = case_kwargs(nx=24, ny=20, W=0, tau=0.7, bc="periodic", sigma_max=0.0, q=q)
    with make_solver(kw, "fp64") as s:
        s.init(*wl.uniform(24, 20, 0))
        P = s.export_populations()
        M, rng = s.M, np.random.default_rng(q)
        F = P[:, M:M + 20, M:M + 24] * (1.0 + 0.01 * rng.standard_normal((q, 20, 24)))
        F[q - 1, 3, 4:9] = (-1e-5, 0.0, 1e-13, 1e-300, -0.0)
        G = F[:, (np.arange(20 + 2 * M) - M) % 20][:, :, (np.arange(24 + 2 * M) - M) % 24]
        s.import_populations(G)
        s.step(1)
        got = s.export_populations()[:, M:M + 20, M:M + 24]
    from oracle.equilibrium import bgk, feq, moments
    from oracle.stencil import lattice
    from paper_2504_20169_gb300 import lattice_info
    e, w, r = lattice_info(q)
    f = np.stack([np.roll(F[i], (e[i, 1], e[i, 0]), axis=(0, 1)) for i in range(q)])
    xi = r * e.astype(float)
    ref = bgk(f, feq(*moments(f, xi), xi, w, lattice(q).order), 0.7)
    assert np.max(np.abs(got - ref) / w[:, None, None]) < 1e-12
