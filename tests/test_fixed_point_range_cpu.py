"""The limits of the fixed-point range on the CPU: states just inside are taken, just outside
refused, and nothing overflows on the limits themselves."""
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
    exe = tmp_path_factory.mktemp("range") / "range"
    subprocess.run([cxx, "-std=c++17", "-O2", "-o", str(exe), str(HERE / "fixed_point_range.cpp")],
                   check=True)
    return exe


@pytest.mark.parametrize("q", [37, 17, 9])
def test_limits(program, q):
    """1/2 < rho < 2, |r u|^2 <= 0.7, |T - 1| <= 1/4, each 1e-9 inside and outside, from moments and
    from given fields. At the limits |f_eq| stays below the 2^60 units that the relaxation allows
    (populations are below 2^59). The polynomial's 15 coefficients are off by up to three units of
    2^-58 each, times at most 337 in all for the velocity (3, 1): 1011 units of 2^-58, which the
    weight and the density (below 2) turn into less than 2 * 1011 / 8 = 253 population units of
    2^-55. An overflow would show as 2^60."""
    from paper_2504_20169_gb300 import lattice_info
    _, w, r = lattice_info(q)
    text = " ".join([str(q), repr(float(r))] + [repr(float(v)) for v in w])
    out = subprocess.run([str(program)], input=text, check=True, capture_output=True,
                         text=True).stdout.split("\n")
    inside, tried_in, outside, tried_out = (int(v) for v in out[0].split())
    assert inside == tried_in and outside == 0 and tried_out > 0
    most, worst = (float(v) for v in out[1].split())
    assert most < 2.0 ** 60
    assert worst < 253
