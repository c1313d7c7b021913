"""FP32 rounding inside the V-cycle against 64 bits, on smooth fields in cells of
unequal widths: there a coefficient of the cell's own value that is rounded by itself
does not cancel against those of its neighbours, and the error that stays is smooth.
One V-cycle from zero, levels in the cluster launch (``fused = 1``) against levels with
the second differences of the stage kernels (``fused = 0``).

Tolerance: in both orders a stage adds the same number of roundings of values of the size
of Y; rms sums of that many roundings, and the rounded coefficients that both have, differ
by some tens of percent (factor 1.5).  A rounded coefficient of the cell's own value gives a
factor of 3 and more.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sg():
    import paper_2306_05332_gb300 as sg
    return sg


def _smooth(shape, seed):
    rng = np.random.default_rng(seed)
    out = np.zeros(shape)
    for _ in range(12):
        k = rng.integers(1, 4, size=len(shape))
        part = rng.standard_normal() / float(np.sum(k * k))
        for d, n in enumerate(shape):
            x = (np.arange(n) + 0.5) / n
            part = part * np.sin(np.pi * k[d] * x).reshape([-1 if a == d else 1 for a in range(len(shape))])
        out += part
    return out.astype(np.float32).astype(np.float64)


def _off(a, ref):
    return np.sqrt(np.mean((a - ref) ** 2) / np.mean(ref ** 2))


@pytest.mark.parametrize("shape,bc,hi", [((48, 40, 56), (1, 0, 0), (1.3, 1.0, 1.7)), ((40, 24, 32), (0, 0, 0), (0.9, 1.0, 1.3)),
                                         ((96, 160), (0, 0), (1.0, 0.7))])
@pytest.mark.parametrize("opts", [dict(), dict(rkl_order=1, s_smooth=2, tau_frac=0.75), dict(smoother="gsrb")])
def test_vcycle_in_the_cluster_launch(shape, bc, hi, opts):
    sg = _sg()
    f = _smooth(shape, 6)
    e = {}
    for precision, fused in (("fp64", 0), ("mixed", 0), ("mixed", 1)):
        g = (sg.Grid if len(shape) == 3 else sg.Grid2D)(shape, (0.0,) * len(shape), hi, bc, precision=precision)
        g.set_options(fused=fused, fixed_cycles=1, coarse_tol=0.0, coarse_max_ss=6, **opts)
        g.set_density(f, 1.0)
        g.solve(tol=0.0, check=False)
        e[precision, fused] = g.potential()
    ref = e["fp64", 0]
    assert _off(e["mixed", 1], ref) < 1.5 * _off(e["mixed", 0], ref)


@pytest.mark.parametrize("shape,hi", [((30, 62, 46), (0.6, 1.0, 0.8)), ((56, 40, 72), (1.1, 0.7, 1.3)), ((48, 48, 48), (1.0, 1.0, 1.0))])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("source", [0.0, -30.0])
def test_fused_superstep(shape, hi, order, source):
    # s = 3, the fused super-step against the three stage launches
    sg = _sg()
    u = _smooth(shape, 5)
    f = (source * u * (1.0 + 0.1 * np.random.default_rng(7).standard_normal(shape))).astype(np.float32)
    out = {}
    for precision, fused, t in (("fp64", 0, torch.float64), ("mixed", 0, torch.float32), ("mixed", 1, torch.float32)):
        g = sg.Grid(shape, (0.0, 0.0, 0.0), hi, (0, 0, 0), precision=precision)
        g.set_options(fused=fused)
        o = torch.empty(shape, dtype=t, device="cuda")
        g.op_superstep(0, order, 3, 0.9, torch.tensor(u, dtype=t, device="cuda"), torch.tensor(f, dtype=t, device="cuda"), o)
        out[precision, fused] = o.double().cpu().numpy()
    ref = out["fp64", 0]
    assert _off(out["mixed", 1], ref) < 1.5 * _off(out["mixed", 0], ref)
