"""FP64 Sigma far below and far above the size of the flow, as it decays ahead
of a front: sweeps on stored coefficients (a context's solve) and sweeps that
divide (the allocation-free solve) give the same bits. At rest the source is
exactly 0, so the numerators are of Sigma's own size: subnormal, around the
smallest normal numbers (where the remainder of a quotient underflows), at the
ends of the range in which the quotient takes the remainder step (2^-500 and
2^500), zero in part of the box, and near overflow (whose infinities turn to NaN).
"""
import ctypes as C

import numpy as np
import pytest

from paper_2505_07392_gb300.inputs import OUTFLOW, PERIODIC, Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("exponent", [-1074, -1060, -1030, -1022, -1000, -970, -960, -500, -499, 0, 499, 500, 1020])
def test_quotients_of_every_size(exponent, solver):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build, igr
    build.build()
    nx, ny, nz = 33, 16, 12
    n = (nz, ny, nx)
    case = Case("box", nx, ny, nz, 1.0 / 33, alpha=1.0 / 33 ** 2, sweeps=4,
                bc=(OUTFLOW, OUTFLOW, PERIODIC, PERIODIC, OUTFLOW, OUTFLOW), sigma_solver=solver)
    rng = np.random.Generator(np.random.Philox(17))
    q = np.zeros((5,) + n)
    q[0], q[4] = rng.uniform(0.5, 1.5, size=n), 2.5
    s0 = np.ldexp(rng.uniform(1.0, 4.0, size=n), exponent) * rng.choice([-1.0, 1.0], size=n)
    s0[:, :, 20:] = 0.0
    q, s0 = torch.from_numpy(q).cuda(), torch.from_numpy(s0).cuda()
    for sweeps in (1, 4):
        with igr.Solver(case, "f64") as s:
            a = s.solve_sigma(q, s0.clone(), sweeps)
        b, (cfg, _jets) = s0.clone(), igr.make_config(case, "f64")
        rc = igr.lib().igr_solve_sigma_noalloc(C.byref(cfg), C.c_void_p(q.data_ptr()), C.c_void_p(b.data_ptr()),
                                               sweeps, C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == igr.OK, igr.lib().igr_noalloc_last_error().decode()
        a, b = a.cpu().numpy(), b.cpu().numpy()
        assert np.array_equal(a, b, equal_nan=True), (sweeps, int((a != b).sum()))
