"""What the library's host code asks of the CUDA runtime, with the runtime replaced (fake_cuda.cpp):
its own objects, no GPU. Kernels do nothing there, so only calls and host state are looked at."""
import ctypes as C
import re
import shutil
import subprocess
from pathlib import Path

import pytest

HERE = Path(__file__).parent
STREAM = C.c_void_p(0x77770)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2504_20169_gb300 import _lib, build
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    build.build()
    objs = [Path(build.BUILD) / (Path(s).stem + ".o") for s in build.sources()]
    if not all(o.exists() for o in objs):
        build.build(force=True)
    include = Path(build.nvcc()).resolve().parent.parent / "include"
    out = tmp_path_factory.mktemp("fake") / "liblbm_fake.so"
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                    f"-I{include}", "-o", str(out), str(HERE / "fake_cuda.cpp"), *map(str, objs)],
                   check=True)
    L = C.CDLL(str(out))
    for name, (res, args) in _lib.PROTOTYPES.items():
        getattr(L, name).restype, getattr(L, name).argtypes = res, args
    L.calls.restype = C.c_char_p
    L.set_captured.argtypes = [C.c_void_p]
    return L


def context(lib, prec=0, bc=1):
    from paper_2504_20169_gb300 import _lib
    grid, sig, bp, out = _lib.lbm_grid(24, 20), _lib.lbm_sigma_profile(0.05, 2, 0), \
        _lib.lbm_bc_params(), C.c_void_p()
    bp.rho0 = bp.T0 = 1.0
    assert lib.lbm_create(C.byref(grid), 17, 0.8, 4, C.byref(sig), bc, C.byref(bp), prec, STREAM,
                          C.byref(out)) == 0
    f = (C.c_double * (32 * 28))(*[1.0] * (32 * 28))
    assert lib.lbm_init(out, f, f, f, f, 0) == 0
    return out


def batch(lib, members):
    out = C.c_void_p()
    assert lib.lbm_batch_create(STREAM, C.byref(out)) == 0
    assert lib.lbm_batch_set(out, (C.c_void_p * len(members))(*[m.value for m in members]),
                             len(members)) == 0
    return out


def steps_of(lib, ctx):
    g = (C.c_int64 * 12)()
    assert lib.lbm_geometry(ctx, g) == 0
    return g[7]


def calls(lib, captured=False):
    """Calls since the last time; launches inside a capture are left out unless asked for."""
    s = lib.calls().decode()
    lib.calls_reset()
    return s if captured else re.sub(r"\([^)]*\)", "", s)


@pytest.mark.parametrize("prec", [0, 1])
def test_a_stream_being_captured_is_refused(lib, prec):
    """Steps count on the host and alternate buffers: replayed from a caller's graph they would not
    be the steps that the context has counted. Refused before anything is launched."""
    c, other = context(lib, prec), context(lib, prec)
    b = batch(lib, [other])
    for done in (0, 40):
        if done:
            assert lib.lbm_step(c, done) == 0 and lib.lbm_batch_step(b, done) == 0
        calls(lib)
        lib.set_captured(STREAM)
        for n in (1, 8, 30):
            assert lib.lbm_step(c, n) == 3          # LBM_ECUDA
            assert b"captured" in lib.lbm_last_error(c)
            assert lib.lbm_batch_step(b, n) == 3
        assert lib.lbm_step(c, 0) == 0 and lib.lbm_batch_step(b, 0) == 0
        lib.set_captured(None)
        assert calls(lib, captured=True) == ""
        assert steps_of(lib, c) == steps_of(lib, other) == done
    lib.lbm_batch_destroy(b)
    lib.lbm_destroy(c), lib.lbm_destroy(other)


@pytest.mark.parametrize("prec", [0, 1])
def test_repeated_short_calls_reach_the_graph_of_eight(lib, prec):
    """Calls of 8 to 11 steps, as a study that samples every ten makes them (after twelve calls the
    remainders have graphs of their own as well)."""
    for n in (8, 9, 10, 11):
        c = context(lib, prec)
        for _ in range(12):
            assert lib.lbm_step(c, n) == 0
        calls(lib)
        for _ in range(2):                        # n odd: one call from each buffer
            assert lib.lbm_step(c, n) == 0
            s = calls(lib)
            assert s == "G" * (1 + n - 8), (n, s)
        assert steps_of(lib, c) == 14 * n
        lib.lbm_destroy(c)


@pytest.mark.parametrize("prec", [0, 1])
def test_first_steps_run_while_a_graph_is_built(lib, prec):
    c = context(lib, prec)
    calls(lib)
    assert lib.lbm_step(c, 100) == 0
    s = calls(lib)
    per_step = s.index("I") // 4                  # four steps launched one by one, then graphs
    assert s == "k" * (4 * per_step) + "I" + 12 * "G", s
    lib.lbm_destroy(c)


@pytest.mark.parametrize("steps", [1, 2, 5, 8, 11])
def test_autotune_times_steps_alone(lib, steps):
    """Nothing is built between the two events around a candidate's timed steps."""
    c = context(lib, 1)
    b = batch(lib, [c])
    calls(lib)
    assert lib.lbm_batch_autotune(b, steps, None, None) == 0
    regions = re.findall(r"R([^RT]*)RT", calls(lib))
    assert regions == ["G" * (steps // 8 + steps % 8)] * 8, regions
    assert steps_of(lib, c) == 8 * (steps + 1)
    lib.lbm_batch_destroy(b)
    lib.lbm_destroy(c)


def test_a_batch_builds_its_graph_behind_running_steps(lib):
    """After a change of members the first steps are launched one by one, and a chunk of a hundred
    steps builds one graph."""
    c, d = context(lib, 1), context(lib, 1)
    b = batch(lib, [c])
    for members in ([c], [c, d]):
        assert lib.lbm_batch_set(b, (C.c_void_p * len(members))(*[m.value for m in members]),
                                 len(members)) == 0
        calls(lib)
        assert lib.lbm_batch_step(b, 100) == 0
        s = calls(lib)
        per_step = s.index("I") // 4
        assert per_step > 0 and s == "k" * (4 * per_step) + "I" + "G" * 12, s
        assert lib.lbm_batch_step(b, 1) == 0
        assert calls(lib) == "k" * per_step
        assert lib.lbm_batch_step(b, 9) == 0      # from the other buffer
        assert calls(lib) == "IG" + "k" * per_step
    assert (steps_of(lib, c), steps_of(lib, d)) == (220, 110)
    lib.lbm_batch_destroy(b)
    lib.lbm_destroy(c), lib.lbm_destroy(d)
