"""FP64 sweeps from stored coefficients (a context's solve) against the sweeps
without them (the allocation-free solve): one sequence of rounded operations,
so the same bits, over odd rows, rows of one block and of several, the
smallest box, every kind of edge, both solvers; and infinities and NaN, which
give the same value or a NaN in both.
"""
import ctypes as C

import numpy as np
import pytest

from paper_2505_07392_gb300.inputs import OUTFLOW, PERIODIC, Case

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 4), (5, 7, 4), (6, 4, 10), (33, 9, 6), (48, 22, 12), (255, 5, 5), (260, 8, 4), (514, 6, 6)]


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


def _both(shape, kind, solver, sweeps, values=()):
    import torch
    from paper_2505_07392_gb300 import igr
    bc = {"periodic": (PERIODIC,) * 6, "outflow": (OUTFLOW,) * 6,
          "mixed": (PERIODIC, PERIODIC, OUTFLOW, OUTFLOW, PERIODIC, PERIODIC)}[kind]
    dx = 1.0 / max(shape)
    case = Case("box", *shape, dx, alpha=dx * dx, sweeps=sweeps, bc=bc, sigma_solver=solver)
    rng = np.random.Generator(np.random.Philox(11))
    n = shape[::-1]
    rho = rng.uniform(0.5, 1.5, size=n)
    q = np.stack([rho] + [rho * rng.uniform(-1, 1, size=n) for _ in range(3)] + [rng.uniform(3, 4, size=n)])
    s0 = rng.uniform(-0.05, 0.05, size=n)
    for (at, v) in values:
        s0.reshape(-1)[at] = v
    q, s0 = torch.from_numpy(q).cuda(), torch.from_numpy(s0).cuda()
    with igr.Solver(case, "f64") as s:
        a = s.solve_sigma(q, s0.clone(), sweeps)
    b, (cfg, _jets) = s0.clone(), igr.make_config(case, "f64")
    rc = igr.lib().igr_solve_sigma_noalloc(C.byref(cfg), C.c_void_p(q.data_ptr()), C.c_void_p(b.data_ptr()), sweeps,
                                           C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == igr.OK, igr.lib().igr_noalloc_last_error().decode()
    return a.cpu().numpy(), b.cpu().numpy()


@pytest.mark.parametrize("kind", ["periodic", "outflow", "mixed"])
@pytest.mark.parametrize("shape", SHAPES)
def test_stored_coefficients_give_the_same_bits(shape, kind):
    bcs = {"periodic": (1, 1, 1), "outflow": (0, 0, 0), "mixed": (1, 0, 1)}[kind]
    even = all(n % 2 == 0 for n, p in zip(shape, bcs) if p)
    for solver in (0, 1) if even else (0,):
        for sweeps in (1, 2, 5):
            a, b = _both(shape, kind, solver, sweeps)
            assert np.array_equal(a, b), (solver, sweeps, np.abs(a - b).max())


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e308, 1e-310])
def test_extreme_values(value):
    a, b = _both((12, 6, 6), "outflow", 0, 2, [(0, value), (200, value)])
    assert np.array_equal(a, b, equal_nan=True)
