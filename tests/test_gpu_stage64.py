"""FP64 stages (one super-step) against the oracle where their kernel branches: strips
of two cells and single cells (odd nx, an array off a 16-byte boundary), equal and
unequal h, with and without face data, first, second and later stages of both orders,
z chunks cut unevenly.  And the restriction without its norms against the one with
them.

Tolerance 1e-12 relative in the max norm (the rounding order differs), as for every
FP64 operator.
"""

import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sg():
    import paper_2306_05332_gb300 as sg
    return sg


def _dev(a, offset=0):
    t = torch.empty(a.size + offset, dtype=torch.float64, device="cuda")[offset:].view(a.shape)
    t.copy_(torch.as_tensor(a))
    return t


@pytest.mark.parametrize("shape", [(4, 6, 2), (9, 5, 7), (11, 9, 64), (70, 8, 66), (5, 33, 65)])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 1)])
@pytest.mark.parametrize("cubic", [True, False])
@pytest.mark.parametrize("order,s,offset", [(1, 1, 0), (1, 3, 1), (2, 2, 0), (2, 3, 1), (2, 5, 0)])
def test_superstep(shape, bc, cubic, order, s, offset):
    lo = (0.0, 0.0, 0.0)
    hi = tuple(n * 0.125 for n in shape[::-1]) if cubic else (1.3, 0.7, 1.1)      # 0.125: exactly equal h
    g = _sg().Grid(shape, lo, hi, bc, precision="fp64")
    faces = W.random_faces(shape, 1)
    g.set_boundary(faces)
    u, f = W.random_field(shape, 2), 50.0 * W.random_field(shape, 3)
    out = _dev(np.zeros(shape), offset)
    g.op_superstep(0, order, s, 0.9, _dev(u, offset), _dev(f, offset), out)
    ref = O.rkl_superstep(u, f, O.spacing(shape, lo, hi), bc, faces, order, s, 0.9)
    err = np.max(np.abs(out.cpu().numpy() - ref)) / np.max(np.abs(ref))
    assert err < 1e-12


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("shape,bc", [((16, 24, 20), (0, 0, 0)), ((8, 12, 36), (1, 1, 1))])
def test_vcycle_without_residual_norms(shape, bc, precision, tol):
    # level by level: the V-cycle's restrictions write no norms (and the coarse sums
    # only where every axis is periodic); the oracle's cycles are the reference
    g = _sg().Grid(shape, bc=bc, precision=precision)
    rho = W.random_field(shape, 4)
    g.set_density(rho, 1.0)
    g.set_options(fused=0, fixed_cycles=2, coarse_tol=0.0, coarse_max_ss=6)
    g.solve(tol=0.0)
    opts = O.Options(coarse_tol=0.0, coarse_max_ss=6)
    ref, _ = O.solve(rho, (0, 0, 0), (1, 1, 1), bc, None, 1.0, opts=opts, cycles=2)
    phi = g.potential()
    assert np.linalg.norm(phi - ref) / np.linalg.norm(ref) < tol
