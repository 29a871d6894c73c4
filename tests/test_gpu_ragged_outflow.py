"""Outflow boxes whose rows end inside a block's tile, where the flux kernel
fills the columns past the stencil with the mirrored last ones: every width
around a tile (32 cells) and its halo, inviscid and viscous, both orders,
against the oracle's L(q; Sigma) in FP64 (the tolerance of the parity tests),
and the face warning: none for a sound state, one for a bad cell in any column.
"""
import ctypes as C

import numpy as np
import pytest

import oracle
from paper_2505_07392_gb300.inputs import OUTFLOW, Case

pytestmark = pytest.mark.gpu

WIDTHS = (4, 5, 12, 17, 18, 29, 31, 32, 33, 34, 35, 36, 50, 61, 63, 64, 66, 70)


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


def _fields(n, seed):
    rng = np.random.Generator(np.random.Philox(seed))
    rho = rng.uniform(0.9, 1.1, size=n)
    u = rng.uniform(-0.3, 0.3, size=(3,) + n)
    return np.concatenate([rho[None], rho * u, (2.5 + 0.5 * rho * (u * u).sum(0))[None]]), rng.uniform(0, 0.02, size=n)


@pytest.mark.parametrize("order,mu", [(5, 0.0), (3, 0.0), (5, 1e-3)])
@pytest.mark.parametrize("nx", WIDTHS)
def test_rhs(nx, order, mu):
    import torch
    from paper_2505_07392_gb300 import igr
    n = (7, 9, nx)
    case = Case("box", nx, 9, 7, 1.0 / 16, alpha=1.0 / 256, bc=(OUTFLOW,) * 6, order=order, mu=mu)
    q, s = _fields(n, nx)
    ref = oracle.rhs(case, q, s)
    for precision, tol in (("f64", 1e-12), ("f32", 1e-4)):
        t = igr.storage_torch_dtype(precision)
        with igr.Solver(case, precision) as sol:
            got = sol.rhs(torch.from_numpy(q).to(t).cuda(), torch.from_numpy(s).to(t).cuda()).double().cpu().numpy()
            assert sol.flags() == 0
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref), precision


@pytest.mark.parametrize("precision", ["f32", "f16", "f16inc"])
def test_face_warning(precision):
    import torch
    from paper_2505_07392_gb300 import igr
    for nx in (5, 30, 34, 61):
        n = (5, 6, nx)
        case = Case("box", nx, 6, 5, 1.0 / 16, alpha=1.0 / 256, bc=(OUTFLOW,) * 6)
        q, s = _fields(n, nx)
        st, qt = igr.storage_torch_dtype(precision), igr.state_torch_dtype(precision)
        s = torch.from_numpy(s).to(st).cuda()
        with igr.Solver(case, precision) as sol:
            for i in {0, nx // 2, nx - 4, nx - 1}:
                b = q.copy()
                b[4, 2, 3, i] = -1.0  # negative pressure in one cell
                sol.rhs(torch.from_numpy(q).to(qt).cuda(), s)
                assert sol.flags() == 0
                sol.rhs(torch.from_numpy(b).to(qt).cuda(), s)
                f = C.c_int()  # (the root of a negative number is reported as well, by the status)
                igr.lib().igr_get_flags(sol.h, C.byref(f))
                assert f.value & 2, (nx, i)
