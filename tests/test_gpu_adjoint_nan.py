"""A NaN in the adjoint at the inflow face reaches the jets' gradients wherever
it lies: here 30 cells and more from the jet, whose profile is 0 there. (It
spreads by at most five cells per stage: three by the faces, one by the sweep,
one by the source.)"""
import math

import numpy as np
import pytest

from paper_2505_07392_gb300.inputs import INFLOW, OUTFLOW, Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_nan_far_from_the_jet(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build, igr
    build.build()
    nx, ny, nz = 72, 12, 8
    dx = 1.0 / nx
    case = Case("jet", nx, ny, nz, dx, alpha=dx * dx, sweeps=1, bc=(OUTFLOW,) * 4 + (INFLOW, OUTFLOW),
                jets=[(8 * dx, 6 * dx, 2 * dx, 1.0, 1.9, 2.0, 1.0)])
    ct = igr.compute_torch_dtype(precision)
    q = torch.zeros((5, nz, ny, nx), dtype=ct, device="cuda")
    q[0], q[3], q[4] = 1.0, 0.3, 2.545
    s0 = torch.zeros((nz, ny, nx), dtype=ct, device="cuda")
    lam = torch.from_numpy(np.random.Generator(np.random.Philox(2)).normal(size=q.shape)).to(ct).cuda()
    with igr.Solver(case, precision) as s:
        assert math.isfinite(s.adjoint_step(q, s0, lam, s0, 0.1 * dx)[2][0])
        lam[3, 0, 6, 70] = math.nan
        lq, _, gw = s.adjoint_step(q, s0, lam, s0, 0.1 * dx)
        assert torch.isfinite(lq[:, :, :, :50]).all()  # the jet's own cells know nothing of it
        assert math.isnan(gw[0])
