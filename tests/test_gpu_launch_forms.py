"""igr_set_kernel_forms selects the kernels that a context's steps launch:
pairs for 0, quads for 1, and by default quads where rows are a multiple of 4
cells (igr_get_launch_forms); the autotuner leaves one of the two set. Whole
steps give the same bits under both, with increments and a jet face, where the
Sigma solve on its own cannot go (stages 2 and 3 read increments)."""
import pytest

from paper_2505_07392_gb300 import inputs
from paper_2505_07392_gb300.inputs import INFLOW, OUTFLOW, Case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


def _jets(nx, ny, nz):
    dx = 1.0 / max(nx, ny, nz)
    return Case("jets", nx, ny, nz, dx, alpha=dx * dx, sweeps=3, bc=(OUTFLOW,) * 4 + (INFLOW, OUTFLOW),
                jets=[(0.4 * nx * dx, 0.5 * ny * dx, 3 * dx, 1.0, 3.0, 2.0, 1.0)])


@pytest.mark.parametrize("precision", ["f64", "f32", "f16inc"])
def test_the_setting_selects(precision):
    import torch
    from paper_2505_07392_gb300 import igr
    sweeps = (lambda form: -1) if precision == "f64" else (lambda form: form)  # FP64 sweeps have one form
    for nx in (36, 64, 128, 130):
        case = _jets(nx, 12, 8)
        q = torch.from_numpy(inputs.jet_initial_state(case)).to(igr.state_torch_dtype(precision)).cuda()
        quads = int(nx % 4 == 0)
        with igr.Solver(case, precision) as s:
            assert s.launch_forms() == (quads, sweeps(quads))
            s.set_kernel_forms(0, 0)
            assert s.launch_forms() == (0, sweeps(0))
            if quads:
                s.set_kernel_forms(1, 0)
                assert s.launch_forms() == (1, sweeps(0))
                s.set_kernel_forms(0, 1)
                assert s.launch_forms() == (0, sweeps(1))
            s.set_kernel_forms(-1, -1)
            assert s.launch_forms() == (quads, sweeps(quads))
            s.set_state(q)
            s.autotune(reps=1)
            assert s.kernel_forms()[0] == s.launch_forms()[0]


@pytest.mark.parametrize("precision", ["f32", "f16", "bf16", "f16inc", "bf16inc"])
@pytest.mark.parametrize("shape", [(36, 13, 9), (64, 20, 12), (128, 16, 8), (260, 9, 6)])
def test_whole_steps_at_tile_edges(shape, precision):
    import torch
    from dataclasses import replace
    from paper_2505_07392_gb300 import igr
    for case in (_jets(*shape), replace(_jets(*shape), sigma_solver=1, mu=1e-3)):
        q = torch.from_numpy(inputs.jet_initial_state(case)).to(igr.state_torch_dtype(precision)).cuda()
        got = []
        for forms in ((1, 1), (0, 0)):
            with igr.Solver(case, precision) as s:
                s.set_kernel_forms(*forms)
                s.set_state(q)
                s.step(2)
                got.append(s.get_state())
        assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
        assert torch.isfinite(got[0][0].double()).all()
