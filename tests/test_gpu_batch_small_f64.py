"""FP64 batches on either side of the rule that groups the sweeps of small
instances (more than ten of them below 32^3 cells): the bits of lone contexts,
with both solvers, uneven sweep counts and a large instance among them."""
from dataclasses import replace

import pytest

from paper_2505_07392_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 10, 11])
def test_small_instances(count):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build, igr
    build.build()
    cases = [inputs.tgv(32)] + [replace(inputs.tgv(8 + 2 * (i % 5), instance=i), sweeps=3 + i % 3,
                                        sigma_solver=i % 2) for i in range(count)]
    q0 = [torch.from_numpy(inputs.initial_state(c)).cuda() for c in cases]
    torch.cuda.synchronize()
    with igr.Batch(cases, "f64") as b:
        for inst, q in zip(b.instances, q0):
            inst.set_state(q)
        b.step(3, sync=True)
        got = [inst.get_state() for inst in b.instances]
    for c, q, g in zip(cases, q0, got):
        with igr.Solver(c, "f64") as s:
            s.set_state(q)
            s.step(3)
            assert all(torch.equal(x, y) for x, y in zip(s.get_state(), g)), (c.nx, c.sweeps)
