"""The one-thread-per-column super-step (RKL s = 2, 3, FP32) where its plan can go
wrong: tiles that do not divide the level, levels narrower than the halo, extents
that are no multiple of a strip, several z chunks and chunks of one plane, wraps and
reflections on every axis.  Against the oracle (FP32 rounding of a few stages: 5e-5
of the largest value, as in ``test_gpu_ops``) and, to the last bit, against the
kernel with tiles of 14 rows, which runs the same arithmetic per strip.
"""

import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [
    ((4, 4, 4), (0, 0, 0)),             # every cell within the halo of a wall
    ((2, 6, 5), (1, 0, 1)),             # periods shorter than the halo
    ((5, 33, 68), (0, 1, 0)),           # one-plane chunks, a second x tile of one strip
    ((37, 58, 131), (0, 0, 1)),         # ragged strips, scalar stores
    ((66, 30, 256), (1, 1, 0)),
    ((31, 94, 34), (0, 0, 0)),
    ((96, 64, 160), (1, 1, 1)),
]


@pytest.mark.parametrize("shape,bc", SHAPES)
@pytest.mark.parametrize("order,s", [(2, 3), (1, 3), (2, 2), (1, 2)])
@pytest.mark.parametrize("zero", [False, True])
def test_column_superstep(shape, bc, order, s, zero):
    import paper_2306_05332_gb300 as sg

    lo, hi = (0.0, -0.5, 0.25), (1.3, 0.2, 1.35)
    g = sg.Grid(shape, lo, hi, bc, precision="mixed")
    u = np.zeros(shape) if zero else W.random_field(shape, 60).astype(np.float32).astype(np.float64)
    rhs = (50.0 * W.random_field(shape, 61)).astype(np.float32).astype(np.float64)
    du = None if zero else torch.tensor(u, dtype=torch.float32, device="cuda")
    dr = torch.tensor(rhs, dtype=torch.float32, device="cuda")
    out = {}
    for rows in (0, 14):
        g.set_options(tile_rows=rows)
        out[rows] = torch.full(shape, float("nan"), dtype=torch.float32, device="cuda")
        g.op_superstep(0, order, s, 0.9, du, dr, out[rows], homogeneous=True)
    torch.cuda.synchronize()
    ref = O.rkl_superstep(u, rhs, O.spacing(shape, lo, hi), bc, None, order, s, 0.9)
    got = out[0].double().cpu().numpy()
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref)) < 5e-5 * np.max(np.abs(ref))
    assert torch.equal(out[0], out[14])
