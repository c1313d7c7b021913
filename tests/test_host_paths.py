"""What the host does with failures and options, without a GPU: ``sg_host.cu`` linked with
launchers and a CUDA runtime that run nothing (``fake_device.cpp``), through the package's
own binding.
"""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_2306_05332_gb300 as sg
from paper_2306_05332_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
RUNNING, DONE, NOT_CONVERGED, NON_FINITE = 0, 1, 2, 3           # DeviceLoop::status


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("fake")
    include = ["-I", os.path.join(B.ROOT, "include"), "-I", B.CSRC]
    host, fake, so = (str(d / n) for n in ("sg_host.o", "fake_device.o", "libsg_fake.so"))
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    for cmd in ([B.nvcc(), *B.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", *include,
                 "-c", os.path.join(B.CSRC, "sg_host.cu"), "-o", host],
                ["g++", "-O1", "-std=c++17", "-fPIC", "-w", *include, "-I", cuda,
                 "-c", os.path.join(HERE, "fake_device.cpp"), "-o", fake],
                ["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", so, host, fake, "-lpthread"]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(so)
    for name, (args, res) in sg._SIGS.items():
        getattr(L, name).argtypes, getattr(L, name).restype = args, res
    L.fake_norm.argtypes = [ctypes.c_double]
    L.fake_loop.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_double]
    return L


@pytest.fixture
def fake(fake_lib, monkeypatch):
    monkeypatch.setattr(sg, "_LIB", fake_lib)
    monkeypatch.setattr(sg, "_torch", lambda: None)
    fake_lib.fake_reset()
    return fake_lib


def _grid(shape, precision="mixed", **opts):
    g = sg.Grid(shape, precision=precision)
    if opts:
        g.set_options(**opts)
    g.set_density(np.ones(shape), 1.0)
    return g


def _log(fake, what):
    out = []
    for i in range(fake.fake_log_size()):
        name, v = ctypes.create_string_buffer(16), (ctypes.c_double * 8)()
        fake.fake_log_entry(i, name, v)
        if name.value.decode() == what:
            out.append(list(v))
    return out


@pytest.mark.parametrize("opts,tol,status", [(dict(fixed_cycles=3), 0.0, DONE),
                                             (dict(max_cycles=1), 1e-9, NOT_CONVERGED)])
def test_nan_left_after_the_last_decision_is_reported(fake, opts, tol, status):
    # a launch that gave up a wait: the loop has ended with a finite residual, the
    # potential holds a NaN, so the residual of the potential is one
    g = _grid((32, 32, 32), **opts)
    fake.fake_loop(status, 0, float("nan"))
    fake.fake_waits(0, 1)
    info = g.solve(tol=tol, check=False)
    assert info["status"] == "SG_ERR_NONFINITE"
    assert np.isnan(info["rel_residual"])
    assert b"gave up a bounded wait" in fake.sg_last_error()


@pytest.mark.parametrize("status,pending,sumsq,want", [(DONE, 0, 1.0, "SG_OK"), (NOT_CONVERGED, 0, 1.0, "SG_ERR_NOT_CONVERGED"),
                                                       (RUNNING, 1, 0.0, "SG_OK"), (RUNNING, 1, float("inf"), "SG_ERR_NONFINITE")])
def test_decision_after_the_inner_loop(fake, status, pending, sumsq, want):
    g = _grid((32, 32, 32), fixed_cycles=0 if pending else 3)
    fake.fake_loop(status, pending, sumsq)
    info = g.solve(tol=1e-9, check=False)
    assert info["status"] == want
    if not pending:
        assert info["rel_residual"] == 0.5            # the loop's own, not the confirmation's


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_waits_are_named_in_both_precisions(fake, precision):
    g = _grid((32, 32, 32), precision)
    fake.fake_waits(0, 1)
    fake.fake_loop(NON_FINITE, 0, float("nan"))
    assert g.solve(tol=1e-9, check=False)["status"] == "SG_ERR_NONFINITE"        # in a cycle
    assert b"gave up a bounded wait" in fake.sg_last_error()
    fake.fake_norm(float("nan"))
    assert g.solve(tol=1e-9, check=False)["status"] == "SG_ERR_NONFINITE"        # at the first residual
    assert b"gave up a bounded wait" in fake.sg_last_error()


@pytest.mark.parametrize("nth", [1, 2, 3])
def test_batch_whose_start_fails_leaves_nothing_in_flight_and_keeps_the_guesses(fake, nth):
    # (the first allocations of a batch are its grids' coarse schedules)
    grids = [_grid((16, 16, 16)), _grid((32, 32, 32)), _grid((24, 24, 24))]
    for g in grids:
        g.set_guess(np.zeros(g.shape))
    fake.fake_reset()
    fake.fake_fail_alloc(nth)
    with pytest.raises(sg.SGError):
        sg.solve_batch(grids, tol=1e-9)
    assert fake.fake_busy() == 0
    fake.fake_reset()
    sg.solve_batch(grids, tol=1e-9)
    assert len(_log(fake, "residual")) == 3         # the residual of each guess
    fake.fake_reset()
    sg.solve_batch(grids, tol=1e-9)
    assert len(_log(fake, "residual")) == 0         # a guess is taken once


@pytest.mark.parametrize("s_smooth", [2, 3])
@pytest.mark.parametrize("opts,want", [(dict(), (0, 0)), (dict(tile_rows=14), (14, 0)), (dict(tile_rows=16, staging="tma"), (16, 1))])
def test_first_supersteps_heed_tile_rows_and_staging(fake, s_smooth, opts, want):
    g = _grid((64, 64, 64), fixed_cycles=1, use_graph=0, s_smooth=s_smooth, **opts)
    g.solve(tol=0.0, check=False)
    first = [e for e in _log(fake, "superstep") if e[3] == 1.0]
    assert len(first) == 1 and first[0][0] == 64 ** 3
    assert (first[0][4], first[0][5]) == want


@pytest.mark.parametrize("order", [1, 2])
def test_stage_coefficients_mean_the_same_in_both_precisions(fake, order):
    stages = {}
    for precision in ("fp64", "mixed"):
        g = _grid((8, 8, 8), precision, fixed_cycles=1, use_graph=0, fused=0, rkl_order=order, s_smooth=3, n_pre=1, n_post=0)
        g.solve(tol=0.0, check=False)
        # cells, order, first, tau, mu~_1, mu~_j tau, gamma~_j
        stages[precision] = [e[:7] for e in _log(fake, "stage") if e[0] == 512]
        fake.fake_reset()
    assert len(stages["fp64"]) == 3 and stages["fp64"] == stages["mixed"]
    mut = (ctypes.c_double * 4)()
    ratio = ctypes.c_double()
    fake.sg_plan_stage_coefficients(order, 3, None, None, mut, None, ctypes.byref(ratio))
    tau = 2.0 / (12.0 * 64.0) * ratio.value
    assert [e[3] for e in stages["fp64"]] == pytest.approx([tau] * 3, rel=1e-14)
    assert stages["fp64"][0][4] == mut[1]
    assert [e[5] for e in stages["fp64"][1:]] == pytest.approx([mut[2] * tau, mut[3] * tau], rel=1e-14)
