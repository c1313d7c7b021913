"""FP64 stages on rows where strips of two cells are taken or just not (the checks of
``test_gpu_stage64`` on other row lengths): 100, 128 and 254 cells (as many idle lanes as by
single cells), 66, 96 and 130 (more), and an array off a 16-byte boundary.
"""

import pytest

import test_gpu_stage64 as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [66, 96, 100, 128, 130, 254])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 1)])
@pytest.mark.parametrize("cubic", [True, False])
@pytest.mark.parametrize("order,s,offset", [(1, 3, 0), (2, 3, 0), (2, 5, 0), (2, 3, 1)])
def test_superstep(nx, bc, cubic, order, s, offset):
    S.test_superstep((5, 9, nx), bc, cubic, order, s, offset)
