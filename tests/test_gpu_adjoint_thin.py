"""The FP64 adjoint on rows around the 12 cells up to which its x-faces march
instead of gathering by warps, with every kind of edge, against the oracle's
adjoint; the same bits from run to run."""
import numpy as np
import pytest

import oracle
from paper_2505_07392_gb300.inputs import INFLOW, OUTFLOW, PERIODIC, Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["periodic", "outflow", "jets"])
@pytest.mark.parametrize("nx", [4, 5, 7, 11, 12, 13])
def test_rows_of_few_cells(nx, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build, igr
    build.build()
    ny, nz, dx = 9, 17, 1.0 / 17
    bc = {"periodic": (PERIODIC,) * 6, "outflow": (OUTFLOW,) * 6, "jets": (OUTFLOW,) * 4 + (INFLOW, OUTFLOW)}[kind]
    jets = [(0.4 * nx * dx, 0.6 * ny * dx, 1.3 * dx, 1.0, 1.9, 2.0, 1.0)] if kind == "jets" else []
    case = Case("box", nx, ny, nz, dx, alpha=dx * dx, sweeps=3, bc=bc, jets=jets)
    rng = np.random.Generator(np.random.Philox(nx))
    n = (nz, ny, nx)
    rho = rng.uniform(0.9, 1.1, size=n)
    u = rng.uniform(0.2, 0.4, size=(3,) + n)
    q = np.concatenate([rho[None], rho * u, (2.5 + 0.5 * rho * (u * u).sum(0))[None]])
    s, lq, ls = rng.uniform(0, 0.02, size=n), rng.normal(size=(5,) + n), rng.normal(size=n)
    oq, os_, ow = oracle.adjoint_step(case, q, s, 0.1 * dx, lq, ls)
    args = [torch.from_numpy(a).cuda() for a in (q, s, lq, ls)]
    with igr.Solver(case, "f64") as sol:
        gq, gs, gw = sol.adjoint_step(*args, 0.1 * dx)
        again = sol.adjoint_step(*args, 0.1 * dx)
    assert torch.equal(gq, again[0]) and torch.equal(gs, again[1]) and gw == again[2]
    for got, ref in ((gq, oq), (gs, os_)):
        assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)
    if jets:
        assert np.abs(np.array(gw) - ow).max() <= 1e-10 * max(1e-3, np.abs(ow).max())
