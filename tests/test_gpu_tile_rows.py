"""The super-step with one stage per thread that ``tile_rows`` and ``staging`` ask for, both
tile heights and both ways of staging, against the kernel with one column per thread: the same
arithmetic per strip, so the same bits.
"""

import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bc", [((5, 33, 68), (0, 1, 0)), ((37, 58, 131), (0, 0, 1)), ((40, 48, 128), (1, 0, 0))])
@pytest.mark.parametrize("rows,staging", [(14, "cp_async"), (16, "cp_async"), (16, "tma")])
@pytest.mark.parametrize("order,s", [(2, 3), (1, 2)])
@pytest.mark.parametrize("zero", [False, True])
def test_same_bits(shape, bc, rows, staging, order, s, zero):
    import paper_2306_05332_gb300 as sg

    g = sg.Grid(shape, (0.0, -0.5, 0.25), (1.3, 0.2, 1.35), bc, precision="mixed")
    u, rhs = (torch.tensor(W.random_field(shape, 60 + i), dtype=torch.float32, device="cuda") for i in (0, 1))
    out = [torch.full(shape, float("nan"), dtype=torch.float32, device="cuda") for _ in range(2)]
    for o, opts in zip(out, (dict(tile_rows=0, staging="cp_async"), dict(tile_rows=rows, staging=staging))):
        g.set_options(**opts)
        g.op_superstep(0, order, s, 0.9, None if zero else u, rhs, o, homogeneous=True)
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])
