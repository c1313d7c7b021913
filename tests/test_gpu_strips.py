"""The strip kernels of a mixed cycle (FP64 update, restriction, prolongation) where
their blocks change shape: rows of fewer than, exactly and more than 32 strips, rows
that leave a block's last lanes idle, a two-dimensional grid (no z term).

The recurrence residual after fixed cycles against f - A phi of the potential that the
grid returns.  It carries the FP64 residual exactly up to the rounding of phi; its norm
is of the FP32 copy (truncated: 2^-23 relative) folded in FP32 over at most a few hundred
strips a thread (1e-4 allowed).  A wrong strip, row or ghost leaves it off by the size of
the residual itself.
"""

import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle import sg_oracle_2d as O2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [
    ((8, 8, 4), (0, 0, 0)),
    ((24, 36, 60), (0, 1, 0)),
    ((16, 20, 128), (0, 0, 1)),
    ((20, 12, 132), (0, 0, 0)),
    ((40, 24, 192), (1, 0, 0)),
    ((96, 64, 256), (0, 0, 0)),
    ((36, 60), (0, 0)),
    ((64, 256), (1, 0)),
]


@pytest.mark.parametrize("shape,bc", SHAPES)
@pytest.mark.parametrize("equal_h", [True, False])
def test_recurrence_residual(shape, bc, equal_h):
    import paper_2306_05332_gb300 as sg

    dims = len(shape)
    lo = (0.0, -0.5, 0.25)[:dims]
    ext = [n * (1.0 if equal_h else s) / 64.0 for n, s in zip(shape[::-1], (1.0, 1.3, 0.8))]
    hi = tuple(a + b for a, b in zip(lo, ext))
    g = (sg.Grid if dims == 3 else sg.Grid2D)(shape, lo, hi, bc, precision="mixed")
    rho = W.random_field(shape, 70)
    g.set_options(fixed_cycles=3)
    g.set_density(rho, 1.0)
    info = g.solve(tol=0.0, levels=2, check=False)
    phi = g.potential()
    if dims == 3:
        r = O.residual(phi, rho, O.spacing(shape, lo, hi), bc)
    else:
        r = O2.residual2d(phi, rho, O2.spacing2d(shape, lo, hi), bc)
    want = np.linalg.norm(r) / np.linalg.norm(rho)
    assert want > 1e-7                          # far above the rounding of phi
    assert abs(info["rel_residual"] - want) < 1e-4 * want
