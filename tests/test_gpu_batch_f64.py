"""FP64 batches, whose grouped step runs the sweeps of instances of 32^3 cells
and more on their own stored coefficients and groups the others (both solvers,
uneven sweep counts, odd rows), and a set_state of one instance between steps:
the bits of lone contexts.
"""
from dataclasses import replace

import pytest

from paper_2505_07392_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


@pytest.mark.parametrize("precision", ["f64", "f32", "f16inc"])
def test_steps_after_set_state(precision):
    import torch
    from paper_2505_07392_gb300 import igr
    cases = [inputs.tgv(16, instance=0), replace(inputs.tgv(32, instance=1), sigma_solver=1),
             replace(inputs.tgv(18, instance=2), sweeps=3), replace(inputs.tgv(32, instance=3), nx=33, sweeps=4)]
    dt = igr.state_torch_dtype(precision)
    q0 = [torch.from_numpy(inputs.initial_state(c)).to(dt).cuda() for c in cases]
    torch.cuda.synchronize()
    with igr.Batch(cases, precision) as b:
        for inst, q in zip(b.instances, q0):
            inst.set_state(q)
        b.step(1)
        first = [inst.get_state() for inst in b.instances]
        b.step(2, sync=True)
        b.instances[1].set_state(q0[1])
        b.step(1)
        b.step(2, sync=True)
        got = [inst.get_state() for inst in b.instances]
    for i, (c, q) in enumerate(zip(cases, q0)):
        with igr.Solver(c, precision) as s:
            s.set_state(q)
            s.step(1)
            assert all(torch.equal(x, y) for x, y in zip(s.get_state(), first[i])), c.name
            s.step(2)
            if i == 1:
                s.set_state(q)
            s.step(3)
            assert all(torch.equal(x, y) for x, y in zip(s.get_state(), got[i])), c.name
