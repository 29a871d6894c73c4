"""A grid of millions of planes keeps every launch within the 65535 blocks that
a grid has along z (128 planes per chunk reach 8.3 million): a uniform state at
rest steps and stays as it is."""
import pytest

from paper_2505_07392_gb300.inputs import OUTFLOW, Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz", [(5, 8_300_000), (4, 8_388_000)])
def test_default_chunks_of_a_tall_grid(nx, nz):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build, igr
    build.build()
    case = Case("tall", nx, 4, nz, 1.0, alpha=1.0, sweeps=1, bc=(OUTFLOW,) * 6)
    q = torch.zeros((5, nz, 4, nx), dtype=torch.float16, device="cuda")
    q[0], q[4] = 1.0, 2.5
    with igr.Solver(case, "f16") as s:
        assert all(-(-nz // zc) <= 65535 for zc in s.tiles())
        s.set_state(q)
        s.step(1)
        got, sigma = s.get_state()
    assert torch.equal(got, q) and not sigma.any()
