"""The coarsest-level solver of one block on levels more than 1024 cells long, whose cell
coordinates it packs (``fused = 0``: not the cluster launch), against the oracle: fixed
super-steps (1, 2 and 3 stages), FP32 rounding 5e-5 of the largest value and FP64 1e-12 as in
``test_gpu_ops``.
"""

import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bc", [((2, 2, 1026), (0, 0, 0)), ((2, 1100, 3), (0, 1, 0)), ((1100, 3, 2), (0, 0, 1)),
                                      ((3, 1500, 2), (1, 0, 0)), ((3000, 2, 2), (0, 0, 0)), ((2, 3, 1024), (1, 0, 0))])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_coarse_solve(shape, bc, precision):
    import paper_2306_05332_gb300 as sg

    t = torch.float64 if precision == "fp64" else torch.float32
    hi = tuple(n / 64.0 for n in shape[::-1])
    g = sg.Grid(shape, (0.0, 0.0, 0.0), hi, bc, precision=precision)
    g.set_options(coarse_tol=0.0, coarse_max_ss=3)
    rhs = W.random_field(shape, 9).astype(np.float32).astype(np.float64)
    out = torch.empty(shape, dtype=t, device="cuda")
    assert g.op_coarse_solve(0, torch.tensor(rhs, dtype=t, device="cuda"), out) == 3
    opts = O.Options(coarse_tol=0.0, coarse_max_ss=3)
    ref = O.coarse_solve(rhs, O.spacing(shape, (0.0, 0.0, 0.0), hi), bc, None, opts)
    got = out.double().cpu().numpy()
    assert np.max(np.abs(got - ref)) < (1e-12 if precision == "fp64" else 5e-5) * np.max(np.abs(ref))
