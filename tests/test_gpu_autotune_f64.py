"""The autotuners leave the sweep chunk alone where the sweeps have none (FP64 on
stored coefficients: a lone context, a large batch instance or one of few) and
still choose it for the many small instances of an FP64 batch and in FP32."""
import pytest

from paper_2505_07392_gb300 import inputs

pytestmark = pytest.mark.gpu

CANDIDATES = {4, 8, 16, 32, 64, 128}


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


def test_lone_contexts():
    import torch
    from paper_2505_07392_gb300 import igr
    case = inputs.tgv(24)
    q = torch.from_numpy(inputs.initial_state(case)).cuda()
    for precision in ("f64", "f32"):
        with igr.Solver(case, precision) as s:
            default = s.tiles()[1]
            mark = next(z for z in range(5, 24) if z != default and z not in CANDIDATES)
            s.set_state(q.to(igr.state_torch_dtype(precision)))
            s.set_tiles(mark, mark, mark)
            got = s.autotune(reps=1)
            assert got[0] != mark and got[2] != mark
            assert (got[1] == mark) == (precision == "f64")


def test_batch():
    import torch
    from paper_2505_07392_gb300 import igr
    # more than ten below 32^3 cells: those sweep together, by chunks
    cases = [inputs.tgv(32), inputs.tgv(33, instance=1)] + [inputs.tgv(16, instance=i) for i in range(2, 13)]
    with igr.Batch(cases, "f64") as b:
        for inst, c in zip(b.instances, cases):
            inst.set_state(torch.from_numpy(inputs.initial_state(c)).cuda())
            inst.set_tiles(7, 7, 7)
        torch.cuda.synchronize()
        tiles = b.autotune(reps=1)
        assert tiles[0][1] == 7 and tiles[1][1] == 7 and all(t[1] != 7 for t in tiles[2:])
        b.step(3, sync=True)
    with igr.Batch(cases[:4], "f64") as b:  # few: each sweeps on its own
        for inst, c in zip(b.instances, cases):
            inst.set_state(torch.from_numpy(inputs.initial_state(c)).cuda())
            inst.set_tiles(7, 7, 7)
        torch.cuda.synchronize()
        assert all(t[1] == 7 for t in b.autotune(reps=1))
