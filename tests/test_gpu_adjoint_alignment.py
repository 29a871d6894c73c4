"""igr_adjoint_step on a state that starts one element into its storage: the
kernels that load four values at once may not be given it. Rows of a multiple
of 4 cells (quads, fitted and full tiles) and others; without jets, where the
adjoint gathers in a fixed order, the result is the aligned state's, bit for
bit."""
import numpy as np
import pytest

from paper_2505_07392_gb300.inputs import OUTFLOW, PERIODIC, Case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


def _sliced(t):
    import torch
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = buf[1:]
    v.copy_(t.reshape(-1))
    return v.view(t.shape)


@pytest.mark.parametrize("precision", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", [(4, 4, 4), (33, 6, 5), (36, 9, 6), (64, 10, 7), (128, 16, 6)])
def test_adjoint_of_a_sliced_state(shape, precision):
    import torch
    from paper_2505_07392_gb300 import igr
    nx, ny, nz = shape
    dx = 1.0 / max(shape)
    case = Case("box", nx, ny, nz, dx, alpha=dx * dx, sweeps=3,
                bc=(OUTFLOW, OUTFLOW, PERIODIC, PERIODIC, OUTFLOW, OUTFLOW))
    rng = np.random.Generator(np.random.Philox(3))
    n = (nz, ny, nx)
    rho = rng.uniform(0.9, 1.1, size=n)
    u = rng.uniform(0.2, 0.4, size=(3,) + n)
    q = np.concatenate([rho[None], rho * u, (2.5 + 0.5 * rho * (u * u).sum(0))[None]])
    st, ct = igr.storage_torch_dtype(precision), igr.compute_torch_dtype(precision)
    q, s = torch.from_numpy(q).to(st).cuda(), torch.from_numpy(rng.uniform(0, 0.02, size=n)).to(st).cuda()
    lq, ls = torch.from_numpy(rng.normal(size=(5,) + n)).to(ct).cuda(), torch.from_numpy(rng.normal(size=n)).to(ct).cuda()
    with igr.Solver(case, precision) as sol:
        ref = sol.adjoint_step(q, s, lq, ls, 0.1 * dx)
        got = sol.adjoint_step(_sliced(q), _sliced(s), _sliced(lq), _sliced(ls), 0.1 * dx)
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
