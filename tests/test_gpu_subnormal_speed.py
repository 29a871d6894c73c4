"""The wave speed of a state at rest whose sound speed squared is subnormal in
FP32 arithmetic: a sound speed of its own and not 0, and NaN for a negative
square (the time step then reports the state).

rho 1, m 0, E = +-2e-39, c^2 = 0.56 E = 1.1e-39. E, p = 0.4 E and 1.4 p round
to the subnormal spacing 2^-149 = 1.4e-45, half of it of 8e-40 each, so c^2 is
off by at most 3 * 0.9e-6 and c by half of that, plus the root's own 2^-22.
"""
import math

import pytest

from paper_2505_07392_gb300.inputs import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f16inc", "bf16inc"])
@pytest.mark.parametrize("shape", [(5, 5, 5), (16, 8, 8)])
def test_subnormal_square(shape, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build, igr
    build.build()
    nx, ny, nz = shape
    case = Case("box", nx, ny, nz, 1.0 / 64, alpha=1e-4)
    q = torch.zeros((5, nz, ny, nx), dtype=torch.float32)
    q[0] = 1.0
    with igr.Solver(case, precision) as s:
        q[4] = 2e-39
        s.set_state(q.cuda())
        assert math.isclose(s.dt(), case.cfl * case.dx / math.sqrt(0.56 * 2e-39), rel_tol=2e-6)
        q[4] = -2e-39
        s.set_state(q.cuda())
        assert math.isnan(s.dt())
        with pytest.raises(igr.IGRError):
            s.step(1)
