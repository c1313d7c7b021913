"""The levels that run in one cluster launch against the level-by-level kernels
(``fused = 0``), where the launch takes more than the two coarsest levels: whole
hierarchies (the resident solve, level 0 included), coarse levels whose x extent is
no multiple of four, slabs of one and of two plane pairs, levels whole in one CTA,
in four warps and in one, two-dimensional levels, both smoothers, both precisions,
smoothing counts of zero.

Tolerances.  FP32: the two paths evaluate the same formulas with another rounding
order; the V-cycle's correction differs by FP32 rounding (1e-5 of its norm, as in
``test_gpu_bottom``; a wrong ghost, weight or coefficient gives 1e-3 and more).
FP64: 1e-12.
"""

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LO, HI = (0.0, -0.5, 0.25), (1.3, 0.2, 1.35)
RKL2 = dict(rkl_order=2, s_smooth=3)


def _sg():
    import paper_2306_05332_gb300 as sg
    return sg


def _solve(shape, bc, levels, precision, fused, cycles=2, tol=0.0, **opts):
    sg = _sg()
    two = len(shape) == 2
    g = (sg.Grid2D(shape, LO[:2], HI[:2], bc, precision=precision) if two
         else sg.Grid(shape, LO, HI, bc, precision=precision))
    if any(b == 0 for b in bc):
        if two:
            rng = np.random.default_rng(3)
            g.set_boundary([rng.standard_normal(n) for n in (shape[0], shape[0], shape[1], shape[1])])
        else:
            g.set_boundary(W.random_faces(shape, 3))
    g.set_density(W.random_field(shape, 4), 1.0)
    g.set_options(fused=fused, fixed_cycles=cycles, **opts)
    info = g.solve(tol=tol, levels=levels, check=False)
    return g.potential(), info


def _close(a, b, tol):
    assert np.all(np.isfinite(a))
    return np.linalg.norm(a - b) / np.linalg.norm(b) < tol


CASES = [
    # shape (nz, ny, nx), bc, levels
    ((32, 32, 32), (0, 0, 0), 5),       # resident, 16 CTAs; levels split, whole, four warps, one warp
    ((8, 8, 8), (0, 1, 0), 3),          # resident, one CTA, every level in few warps
    ((4, 4, 4), (0, 0, 0), 2),          # the smallest: one warp throughout
    ((16, 16, 16), (1, 1, 1), 4),       # resident, split, coarse means removed
    ((36, 20, 28), (0, 1, 1), 2),       # coarse x extent 14, 9 CTAs of two plane pairs, z wrap
    ((40, 24, 72), (1, 0, 0), 3),       # coarse x extent 18
    ((72, 40, 56), (0, 0, 1), 3),       # launch from level 1
    ((12, 8, 40), (1, 0, 1), 2),        # few planes: more CTAs than plane pairs on the coarse level
    ((64, 64, 64), (1, 0, 0), 6),
]


@pytest.mark.parametrize("shape,bc,levels", CASES)
@pytest.mark.parametrize("opts", [RKL2, dict(rkl_order=1, s_smooth=2, tau_frac=0.75, n_pre=1, n_post=2),
                                  dict(RKL2, s_smooth=5, n_pre=3, inner_n_pre=0, inner_n_post=2),
                                  dict(smoother="gsrb"), dict(smoother="gsrb", omega=0.0, n_pre=0, n_post=2)])
def test_launch_matches_level_by_level_fp32(shape, bc, levels, opts):
    a, ia = _solve(shape, bc, levels, "mixed", 1, **opts)
    b, ib = _solve(shape, bc, levels, "mixed", 0, **opts)
    if all(x == 1 for x in bc):
        a, b = a - a.mean(), b - b.mean()
    assert _close(a, b, 1e-5)
    assert ia["coarse_ss"] == ib["coarse_ss"] and ia["cycles"] == ib["cycles"] == 2


@pytest.mark.parametrize("shape,bc,levels", [((64, 64, 64), (0, 0, 0), 5), ((48, 32, 40), (1, 0, 0), 3),
                                             ((32, 32, 32), (1, 1, 1), 4), ((16, 16, 16), (0, 1, 0), 4)])
@pytest.mark.parametrize("opts", [RKL2, dict(smoother="gsrb")])
def test_launch_matches_level_by_level_fp64(shape, bc, levels, opts):
    a, ia = _solve(shape, bc, levels, "fp64", 1, coarse_tol=0.0, coarse_max_ss=6, **opts)
    b, ib = _solve(shape, bc, levels, "fp64", 0, coarse_tol=0.0, coarse_max_ss=6, **opts)
    if all(x == 1 for x in bc):
        a, b = a - a.mean(), b - b.mean()
    assert _close(a, b, 1e-12)


@pytest.mark.parametrize("shape,bc", [((128, 96), (0, 0)), ((64, 64), (1, 1)), ((20, 36), (1, 0)), ((256, 64), (0, 1))])
@pytest.mark.parametrize("precision,tol", [("mixed", 1e-5), ("fp64", 1e-12)])
def test_launch_matches_level_by_level_2d(shape, bc, precision, tol):
    # (a fixed number of coarse super-steps: both sides run the same stages)
    kw = dict(RKL2, coarse_tol=0.0, coarse_max_ss=6)
    a, _ = _solve(shape, bc, 0, precision, 1, **kw)
    b, _ = _solve(shape, bc, 0, precision, 0, **kw)
    if all(x == 1 for x in bc):
        a, b = a - a.mean(), b - b.mean()
    assert _close(a, b, tol)


@pytest.mark.parametrize("shape,bc,levels", [((32, 32, 32), (0, 0, 0), 5), ((16, 24, 20), (0, 1, 0), 2)])
def test_resident_solve_takes_the_decisions_of_the_loop_on_the_host(shape, bc, levels):
    # the inner loop in one launch (use_graph = 1) against one launch a cycle with the
    # host's decisions (2): the same arithmetic, so the same potential to the last
    # bit; tolerance, cycle cap and maximum-residual stop
    for kw, tol in ((dict(), 1e-9), (dict(max_cycles=3), 1e-14), (dict(max_residual_tol=1e-4), 0.0)):
        out = {}
        for mode in (1, 2):
            out[mode] = _solve(shape, bc, levels, "mixed", 1, cycles=0, tol=tol, use_graph=mode, **RKL2, **kw)
        (a, ia), (b, ib) = out[1], out[2]
        np.testing.assert_array_equal(a, b)
        assert ia["cycles"] == ib["cycles"] and ia["status"] == ib["status"] and ia["coarse_ss"] == ib["coarse_ss"]
        np.testing.assert_allclose(ia["history"], ib["history"], rtol=1e-5)


def test_resident_solve_reports_a_non_finite_density():
    sg = _sg()
    g = sg.Grid((16, 16, 16), precision="mixed")
    rho = W.random_field((16, 16, 16), 5)
    rho[3, 3, 3] = np.nan
    g.set_density(rho, 1.0)
    assert g.solve(tol=1e-8, check=False)["status"] == "SG_ERR_NONFINITE"
    g.set_density(W.random_field((16, 16, 16), 5), 1.0)
    assert g.solve(tol=1e-8)["status"] == "SG_OK"
