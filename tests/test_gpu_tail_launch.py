"""Which levels the cluster launch takes, by the launches of a cycle (the comparisons with the
level-by-level kernels in ``test_gpu_tail`` would also pass if it were never chosen), and a
thin two-dimensional level whose slabs' owners are found by the largest quotients.
"""

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _launches_per_cycle(shape, levels, precision, fused, **opts):
    import paper_2306_05332_gb300 as sg
    n = {}
    for cycles in (2, 5):
        g = (sg.Grid if len(shape) == 3 else sg.Grid2D)(shape, precision=precision)
        g.set_density(W.random_field(shape, 4), 1.0)
        g.set_options(fused=fused, fixed_cycles=cycles, **opts)
        n[cycles] = g.solve(tol=0.0, levels=levels, check=False)["kernel_launches"]
    assert (n[5] - n[2]) % 3 == 0
    return (n[5] - n[2]) // 3


# shape, levels, options, launches of a cycle: resident 0; from level 1 the smoothing of level 0
# (3 column super-steps; GS-RB 6 colours), its restriction, the launch, prolongation,
# update and the loop's step; the launch from level 2 also level 1 by stages
@pytest.mark.parametrize("shape,levels,opts,want", [
    ((32, 32, 32), 5, dict(), 0),
    ((8, 8, 8), 3, dict(), 0),
    ((4, 4, 4), 2, dict(), 0),
    ((16, 16, 16), 4, dict(smoother="gsrb"), 0),
    ((32, 24, 32), 3, dict(s_smooth=5, n_pre=3), 0),
    ((128, 96), 0, dict(), 0),
    ((72, 40, 56), 3, dict(), 8),
    ((64, 64, 64), 6, dict(), 8),
    ((64, 64, 64), 6, dict(smoother="gsrb"), 11),
    ((64, 64, 128), 4, dict(), 8 + 2 + 9),
])
def test_mixed(shape, levels, opts, want):
    assert _launches_per_cycle(shape, levels, "mixed", 1, **opts) == want
    assert _launches_per_cycle(shape, levels, "mixed", 0, **opts) > want


@pytest.mark.parametrize("shape,levels,stages", [((64, 64, 64), 5, 2), ((32, 32, 32), 4, 1), ((16, 16, 16), 4, 1)])
def test_fp64(shape, levels, stages):
    # `stages` levels by nine stages, restriction and prolongation each; the launch, the
    # residual and the loop's step
    assert _launches_per_cycle(shape, levels, "fp64", 1) == 11 * stages + 3
    assert _launches_per_cycle(shape, levels, "fp64", 0) > 11 * stages + 3


def test_thin_level():
    # 4 x 8192 cells: 4096 plane pairs over 16 CTAs (tolerance as in test_gpu_tail)
    import paper_2306_05332_gb300 as sg
    shape = (8192, 4)
    out = {}
    for fused in (0, 1):
        g = sg.Grid2D(shape, (0.0, 0.0), (1.0, 2048.0), (0, 0), precision="mixed")
        g.set_density(W.random_field(shape, 4), 1.0)
        g.set_options(fused=fused, fixed_cycles=2, coarse_tol=0.0, coarse_max_ss=3)
        g.solve(tol=0.0, check=False)
        out[fused] = g.potential()
    assert _launches_per_cycle(shape, 0, "mixed", 1, coarse_tol=0.0, coarse_max_ss=3) == 0
    assert np.linalg.norm(out[1] - out[0]) < 1e-5 * np.linalg.norm(out[0])


def test_resident_solves_from_several_threads():
    # a grid and a stream per host thread; each solve's potential is what it is alone
    import threading

    import paper_2306_05332_gb300 as sg

    shapes = [(32, 32, 32), (16, 24, 20), (128, 96), (16, 16, 16)]

    def solve(i, out, barrier=None):
        stream = torch.cuda.Stream()
        make = sg.Grid if len(shapes[i]) == 3 else sg.Grid2D
        g = make(shapes[i], precision="mixed", stream=stream.cuda_stream)
        g.set_density(W.random_field(shapes[i], i), 1.0)
        if barrier:
            barrier.wait()
        for _ in range(3):
            g.solve(tol=1e-9)
        out[i] = g.potential()

    alone, together = {}, {}
    for i in range(len(shapes)):
        solve(i, alone)
    barrier = threading.Barrier(len(shapes), timeout=60)
    threads = [threading.Thread(target=solve, args=(i, together, barrier)) for i in range(len(shapes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(len(shapes)):
        np.testing.assert_array_equal(together[i], alone[i])
