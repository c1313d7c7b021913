"""FP32 restriction and prolongation on strips where their blocks change shape: rows just
above, at and below a sixth of idle lanes, one lane idle, one strip past a block.  Against the
oracle, FP32 rounding of a few operations (5e-5 of the largest value, as in ``test_gpu_ops``).
"""

import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.tensor(a, dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("nx", [104, 108, 124, 132, 316, 320])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 1)])
def test_transfers(nx, bc):
    import paper_2306_05332_gb300 as sg

    shape, lo, hi = (8, 24, nx), (0.0, -0.5, 0.25), (1.3, 0.2, 1.35)
    g = sg.Grid(shape, lo, hi, bc, precision="mixed")
    u, rhs = (W.random_field(shape, 14 + i).astype(np.float32).astype(np.float64) for i in (0, 1))
    coarse = torch.full(tuple(n // 2 for n in shape), float("nan"), dtype=torch.float32, device="cuda")
    g.op_residual_restrict(0, _dev(u), _dev(rhs), coarse, homogeneous=True)
    ref = O.restrict(-O.residual(u, rhs, O.spacing(shape, lo, hi), bc, None))
    assert np.max(np.abs(coarse.double().cpu().numpy() - ref)) < 5e-5 * np.max(np.abs(ref))
    c = W.random_field(tuple(n // 2 for n in shape), 17).astype(np.float32).astype(np.float64)
    fine = _dev(u)
    g.op_prolong_correct(0, _dev(c), fine)
    ref = u + O.prolong(c, bc)
    assert np.max(np.abs(fine.double().cpu().numpy() - ref)) < 5e-5 * np.max(np.abs(ref))
