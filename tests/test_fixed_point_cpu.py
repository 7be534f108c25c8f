"""The fixed-point form of the FP64 node update on the CPU: no less exact than double arithmetic
over its range (both against long double), and refused outside it."""
import shutil
import subprocess
from pathlib import Path

import pytest

HERE = Path(__file__).parent


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    exe = tmp_path_factory.mktemp("fixed") / "check"
    subprocess.run([cxx, "-std=c++17", "-O2", "-o", str(exe), str(HERE / "fixed_point_check.cpp")],
                   check=True)
    return exe


def check(program, q, args):
    from paper_2504_20169_gb300 import lattice_info
    _, w, r = lattice_info(q)
    text = " ".join([str(q), repr(float(r))] + [repr(float(v)) for v in w])
    out = subprocess.run([str(program)] + [str(a) for a in args], input=text, check=True,
                         capture_output=True, text=True).stdout.split()
    taken, tried = int(out[0]), int(out[1])
    v = [float(x) for x in out[2:]]
    return taken, tried, v[:4], v[4:]


# speed, |T - 1|, density range, noise, omega
RANGES = [(0.02, 0.001, 0.999, 1.001, 1e-4, 1.25), (0.3, 0.02, 0.95, 1.05, 1e-3, 1 / 0.55),
          (0.28, 0.2, 0.55, 1.3, 0.02, 1.9), (0.2, 0.05, 3.8, 4.2, 0.01, 0.7),
          (0.48, 0.24, 0.6, 1.3, 0.01, 1.0)]


@pytest.mark.parametrize("q", [37, 17, 9])
@pytest.mark.parametrize("args", RANGES)
def test_no_less_exact_than_double(program, q, args):
    """Root mean square errors of populations, rho, u and T after one collision. The last rounding
    (to double) is common to both, so equality is the floor; 10 % covers the sampling. At the faster
    and hotter ends many nodes have a negative population (D2Q17's third-order equilibrium first)
    and are refused."""
    taken, tried, double, fixed = check(program, q, args)
    assert taken > 0.1 * tried
    for d, f in zip(double, fixed):
        assert f <= 1.1 * d


@pytest.mark.parametrize("q", [37, 17, 9])
@pytest.mark.parametrize("args", [(0.1, 0.001, 2.6, 2.7, 1e-3, 1.0), (1e-3, 0.001, 1.0, 1.0, 2.5, 1.0)])
def test_out_of_range_is_refused(program, q, args):
    """Densities at 2.65 = 0.66 of the scale 4 are taken (the exponent follows the mean density);
    noise above 1 makes populations negative: those nodes go to the FP64 arithmetic."""
    taken, tried, _, _ = check(program, q, args)
    assert taken == tried if args[4] < 1 else taken < 0.1 * tried
