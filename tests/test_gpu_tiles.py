"""The two forms of the source and sweep kernels at the edges of their tiles.

Rows of a multiple of 4 cells and aligned buffers take quads (4-wide
accesses, tiles fitted to the row, or the full tile with one or two rows per
thread); a buffer sliced one element into its storage takes pairs (element
accesses). Both evaluate one sequence of rounded operations, so the Sigma
solve gives the same bits; in FP64 both are the oracle's to 1e-12.
"""
import numpy as np
import pytest

import oracle
from paper_2505_07392_gb300.inputs import OUTFLOW, PERIODIC, Case

pytestmark = pytest.mark.gpu

# one tile, one quad more or less, several tiles, rows and planes that cut a
# tile, the smallest box
SHAPES = [(4, 4, 4), (12, 5, 6), (16, 33, 5), (32, 7, 9), (48, 21, 13), (96, 11, 8), (124, 9, 7), (128, 8, 5),
          (128, 16, 6), (132, 17, 6), (260, 9, 5)]


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
    bc = {"periodic": (PERIODIC,) * 6, "outflow": (OUTFLOW,) * 6,
          "mixed": (PERIODIC, PERIODIC, OUTFLOW, OUTFLOW, PERIODIC, PERIODIC)}[kind]
    dx = 1.0 / max(shape)
    return Case("box", nx, ny, nz, dx, alpha=dx * dx, sweeps=3, bc=bc)


def _fields(case, seed):
    rng = np.random.Generator(np.random.Philox(seed))
    n = (case.nz, case.ny, case.nx)
    rho = rng.uniform(0.5, 1.5, size=n)
    q = np.stack([rho] + [rho * rng.uniform(-1, 1, size=n) for _ in range(3)] + [rng.uniform(3, 4, size=n)])
    return q, rng.uniform(-0.05, 0.05, size=n)


def _sliced(t):
    import torch
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = buf[1:]
    v.copy_(t.reshape(-1))
    return v.view(t.shape)


@pytest.mark.parametrize("kind", ["periodic", "outflow", "mixed"])
@pytest.mark.parametrize("shape", SHAPES)
def test_quads_equal_pairs(shape, kind):
    import torch
    from dataclasses import replace
    from paper_2505_07392_gb300 import igr
    case = _case(shape, kind)
    q64, s64 = _fields(case, 3)
    red_black = all(n % 2 == 0 for n, b in zip(shape, case.bc[::2]) if b == PERIODIC)
    for precision in ("f64", "f32", "f16", "bf16"):
        dt = igr.storage_torch_dtype(precision)
        q, s0 = torch.from_numpy(q64).to(dt).cuda(), torch.from_numpy(s64).to(dt).cuda()
        for solver in (0, 1) if red_black else (0,):
            for tiles in (None, (4, 4, 4)):
                with igr.Solver(replace(case, sigma_solver=solver), precision) as s:
                    if tiles:
                        s.set_tiles(*tiles)
                    a = s.solve_sigma(q, s0.clone(), 3)
                    b = s.solve_sigma(_sliced(q), _sliced(s0), 3)
                    assert torch.equal(a, b), (precision, solver, tiles)
                    if precision == "f64" and solver == 0:
                        ref = oracle.jacobi(case, q64, oracle.source(case, q64), s64, 3)
                        assert np.abs(a.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


def test_two_rows_per_thread_equal_pairs():
    """16-bit storage, full tiles, 16M cells: the sweep with two rows per thread."""
    import torch
    from paper_2505_07392_gb300 import igr
    case = _case((256, 512, 128), "mixed")
    g = torch.Generator(device="cuda").manual_seed(5)
    n = (case.nz, case.ny, case.nx)
    q = torch.rand((5,) + n, generator=g, device="cuda").add_(0.5).half()
    s0 = torch.rand(n, generator=g, device="cuda").mul_(0.05).half()
    with igr.Solver(case, "f16") as s:
        assert torch.equal(s.solve_sigma(q, s0.clone(), 3), s.solve_sigma(_sliced(q), _sliced(s0), 3))
