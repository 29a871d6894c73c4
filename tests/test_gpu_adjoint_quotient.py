"""mu = lambda / D of the reversed sweeps is the rounded quotient.

At rest with rho = 1 and Sigma = 0 on a periodic box, a sweep's reverse sends
mu beta to each of the six neighbours, D = 1 + 6 beta everywhere, and nothing
else reaches Sigma's adjoint (dt is far below the last place). One sweep in
each of the three stages takes a single value v to the cell three to the right
along one path only: with beta a power of two the result is exactly
beta^3 times three quotients by D, each rounded to nearest.
"""
import numpy as np
import pytest

from paper_2505_07392_gb300.inputs import PERIODIC, Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta", [0.25, 1.0, 2.0])
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_three_quotients(precision, beta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build, igr
    build.build()
    N, dx = 48, 0.125
    case = Case("box", N, N, N, dx, alpha=beta * dx * dx, sweeps=1, bc=(PERIODIC,) * 6)
    t = igr.storage_torch_dtype(precision)
    num = np.float64 if precision == "f64" else np.float32
    q = torch.zeros((5, N, N, N), dtype=t, device="cuda")
    q[0], q[4] = 1.0, 2.5
    zero = torch.zeros((N, N, N), dtype=t, device="cuda")
    v = np.random.Generator(np.random.Philox(23)).uniform(-4.0, 4.0, size=(6, 6, 6)).astype(num)
    lam = np.zeros((N, N, N), dtype=num)
    lam[::8, ::8, ::8] = v
    with igr.Solver(case, precision) as s:
        _, got, _ = s.adjoint_step(q, zero, torch.zeros_like(q), torch.from_numpy(lam).cuda(), 1e-300)
    want = v
    for _ in range(3):
        want = num(beta) * (want / num(1 + 6 * beta))
    assert np.array_equal(got.cpu().numpy()[::8, ::8, 3::8], want)
