"""The adjoint kernels at the edges of their segments and chunks: rows around
the 27 cells that a warp gathers, short and long marches, boxes of the
smallest size, every boundary kind; against the oracle's FP64 adjoint, and
the same bits from run to run where the kernels gather."""
import numpy as np
import pytest

import oracle
from paper_2505_07392_gb300.inputs import INFLOW, OUTFLOW, PERIODIC, Case

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 4), (5, 27, 6), (21, 5, 9), (22, 8, 5), (27, 6, 11), (28, 13, 4), (48, 7, 5), (55, 4, 8),
          (6, 9, 41)]


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


def _case(shape, kind):
    nx, ny, nz = shape
    dx = 1.0 / max(shape)
    bc = {"periodic": (PERIODIC,) * 6, "outflow": (OUTFLOW,) * 6,
          "mixed": (PERIODIC, PERIODIC, OUTFLOW, OUTFLOW, PERIODIC, PERIODIC),
          "jets": (OUTFLOW, OUTFLOW, PERIODIC, PERIODIC, INFLOW, OUTFLOW)}[kind]
    jets = [(0.4 * nx * dx, 0.6 * ny * dx, 1.3 * dx, 1.0, 1.9, 2.0, 1.0),
            (0.8 * nx * dx, 0.3 * ny * dx, 1.1 * dx, 0.9, 1.4, 1.8, 2.0)] if kind == "jets" else []
    return Case("box", nx, ny, nz, dx, alpha=dx * dx, sweeps=3, bc=bc, jets=jets)


def _inputs(case, seed):
    rng = np.random.Generator(np.random.Philox(seed))
    n = (case.nz, case.ny, case.nx)
    rho = rng.uniform(0.9, 1.1, size=n)
    u = rng.uniform(0.2, 0.4, size=(3,) + n)
    q = np.concatenate([rho[None], rho * u, (2.5 + 0.5 * rho * (u * u).sum(0) + rng.uniform(0, 0.1, size=n))[None]])
    return q, rng.uniform(0, 0.02, size=n), rng.normal(size=(5,) + n), rng.normal(size=n)


@pytest.mark.parametrize("kind", ["periodic", "outflow", "mixed", "jets"])
@pytest.mark.parametrize("shape", SHAPES)
def test_adjoint_step_at_tile_edges(shape, kind):
    import torch
    from paper_2505_07392_gb300 import igr
    case = _case(shape, kind)
    q, s, lq, ls = _inputs(case, 7)
    dt = 0.1 * case.dx
    oq, os_, ow = oracle.adjoint_step(case, q, s, dt, lq, ls)
    for precision, tol in (("f64", 1e-10), ("f32", 1e-4)):
        t = igr.storage_torch_dtype(precision)
        args = [torch.from_numpy(a).to(t).cuda() for a in (q, s, lq, ls)]
        with igr.Solver(case, precision) as sol:
            gq, gs, gw = sol.adjoint_step(*args, dt)
            again = sol.adjoint_step(*args, dt)
        if precision == "f64" or not case.jets:  # gathered: deterministic
            assert torch.equal(gq, again[0]) and torch.equal(gs, again[1]) and gw == again[2]
        for got, ref in ((gq, oq), (gs, os_)):
            err = np.linalg.norm(got.double().cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= tol, (precision, err)
        if case.jets:
            assert np.abs(np.array(gw) - ow).max() <= tol * max(1e-3, np.abs(ow).max()), precision
