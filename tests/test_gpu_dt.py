"""dt = cfl dx / max(|u| + c) where the wave-speed kernel changes form: four
cells per load (n a multiple of 4) or one, one warp or many in the final
reduction, the fastest cell first, last and next to a block's edge.

One fastest cell (rho 1, m (3, 0, 0), E 7, so |u| 3, p 1, c sqrt 1.4); every
other cell is at rest with a lower sound speed. Tolerance: a handful of
roundings of numbers of the size of E, over a speed of 4.2: 16 units in the
last place.
"""
import math

import pytest

from paper_2505_07392_gb300.inputs import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,eps", [("f64", 2.0**-53), ("f32", 2.0**-24), ("f16", 2.0**-24)])
@pytest.mark.parametrize("shape", [(4, 4, 4), (5, 5, 5), (6, 7, 9), (7, 9, 4), (64, 33, 20), (129, 65, 33), (136, 100, 96)])
def test_dt_of_the_fastest_cell(shape, precision, eps):
    import torch
    from paper_2505_07392_gb300 import igr
    nx, ny, nz = shape
    case = Case("box", nx, ny, nz, 1.0 / 64, alpha=1e-4)
    n = nx * ny * nz
    with igr.Solver(case, precision) as s:
        for at in {0, n - 1, n // 2, min(n - 1, 1023), min(n - 1, 1024)}:
            q = torch.zeros((5, n), dtype=igr.storage_torch_dtype(precision), device="cuda")
            q[0], q[4] = 1.0, 2.0
            q[1, at], q[4, at] = 3.0, 7.0
            s.set_state(q.view(5, nz, ny, nx))
            assert math.isclose(s.dt(), case.cfl * case.dx / (3.0 + math.sqrt(1.4)), rel_tol=16 * eps), at
