"""Full tiles where other tests do not reach them: two rows per thread with
red-black sweeps and every kind of edge, alone and in a batch; the FP64 full
tile, which the allocation-free solve and small FP64 batch instances launch;
and two rows per thread under the bounds-checking build. Quads and pairs
evaluate one sequence of rounded operations, so results are the same bits."""
import ctypes as C
import gc

import pytest

from paper_2505_07392_gb300 import inputs
from paper_2505_07392_gb300.inputs import OUTFLOW, PERIODIC, Case

pytestmark = pytest.mark.gpu

EDGES = {"periodic": (PERIODIC,) * 6, "outflow": (OUTFLOW,) * 6,
         "mixed": (PERIODIC, PERIODIC, OUTFLOW, OUTFLOW, PERIODIC, PERIODIC)}
BIG = (256, 512, 128)  # 2^24 cells: two rows per thread in 16-bit storage


@pytest.fixture(autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_07392_gb300 import build
    build.build()
    yield


def _case(shape, kind, solver, sweeps=3):
    dx = 1.0 / max(shape)
    return Case("box", *shape, dx, alpha=dx * dx, sweeps=sweeps, bc=EDGES[kind], sigma_solver=solver)


def _random(shape, dtype, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = shape[::-1]
    q = torch.rand((5,) + n, generator=g, device="cuda").add_(0.5)
    q[4].add_(3.0)
    return q.to(dtype), torch.rand(n, generator=g, device="cuda").mul_(0.05).to(dtype)


def _sliced(t):
    import torch
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = buf[1:]
    v.copy_(t.reshape(-1))
    return v.view(t.shape)


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("kind", sorted(EDGES))
@pytest.mark.parametrize("precision", ["f16", "bf16"])
def test_two_rows_per_thread(precision, kind, solver):
    import torch
    from paper_2505_07392_gb300 import igr
    q, s0 = _random(BIG, igr.storage_torch_dtype(precision), 5)
    with igr.Solver(_case(BIG, kind, solver), precision) as s:
        assert torch.equal(s.solve_sigma(q, s0.clone(), 3), s.solve_sigma(_sliced(q), _sliced(s0), 3))


@pytest.mark.parametrize("solver", [0, 1])
def test_two_rows_per_thread_in_a_batch(solver):
    """Grouped steps (from the second on) against a lone context of pairs."""
    import torch
    from paper_2505_07392_gb300 import igr
    cases = [_case(BIG, "mixed", solver), _case((128, 16, 8), "mixed", solver)]
    q0 = []
    for i, c in enumerate(cases):
        x = torch.arange(c.nx, device="cuda", dtype=torch.float32) / c.nx
        q = torch.zeros((5, c.nz, c.ny, c.nx), device="cuda")
        q[0] = 1.0 + 0.1 * torch.sin(6.283185 * x)
        q[1], q[2], q[4] = 0.3 * q[0], -0.2 * q[0] * torch.cos(6.283185 * x), 3.0
        q0.append(q)
    torch.cuda.synchronize()
    with igr.Batch(cases, "f16inc") as b:
        for inst, q in zip(b.instances, q0):
            inst.set_state(q)
        b.step(3, sync=True)
        got = [inst.get_state() for inst in b.instances]
    for c, q, g in zip(cases, q0, got):
        with igr.Solver(c, "f16inc") as s:
            s.set_kernel_forms(0, 0)
            s.set_state(q)
            s.step(3)
            assert all(torch.equal(x, y) for x, y in zip(s.get_state(), g)), c.nx


def _noalloc(case, q, s0, sweeps):
    import torch
    from paper_2505_07392_gb300 import igr
    cfg, _jets = igr.make_config(case, "f64")
    rc = igr.lib().igr_solve_sigma_noalloc(C.byref(cfg), C.c_void_p(q.data_ptr()), C.c_void_p(s0.data_ptr()), sweeps,
                                           C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == igr.OK, igr.lib().igr_noalloc_last_error().decode()
    return s0


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("kind", sorted(EDGES))
@pytest.mark.parametrize("shape", [(128, 8, 6), (128, 16, 6), (256, 8, 4), (48, 22, 12), (36, 10, 8)])
def test_fp64_quads_pairs_and_stored_coefficients(shape, kind, solver):
    import torch
    from paper_2505_07392_gb300 import igr
    case = _case(shape, kind, solver)
    q, s0 = _random(shape, torch.float64, 9)
    quads = _noalloc(case, q, s0.clone(), 3)
    pairs = _noalloc(case, _sliced(q), _sliced(s0), 3)
    with igr.Solver(case, "f64") as s:
        stored = s.solve_sigma(q, s0.clone(), 3)
    assert torch.equal(quads, pairs) and torch.equal(quads, stored)


@pytest.mark.parametrize("solver", [0, 1])
def test_fp64_full_tile_in_a_batch(solver):
    import torch
    from dataclasses import replace
    from paper_2505_07392_gb300 import igr
    cases = [replace(inputs.tgv(128, instance=i), ny=8 * i, nz=12 // i, sigma_solver=solver) for i in (1, 2)]
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
            assert all(torch.equal(x, y) for x, y in zip(s.get_state(), g)), c.ny


def test_two_rows_per_thread_in_bounds(monkeypatch):
    from paper_2505_07392_gb300 import build, igr
    path = build.build(debug_bounds=True)
    gc.collect()  # no handle of the normal library may reach the debug one
    monkeypatch.setattr(igr, "LIB_PATH", path)
    monkeypatch.setattr(igr, "_lib", None)  # restored to the normal library afterwards
    h = C.c_ulonglong()
    assert igr.lib().igr_debug_bounds_hits(C.byref(h), 1) == igr.OK
    q, s0 = _random(BIG, igr.storage_torch_dtype("f16"), 5)
    for solver in (0, 1):
        for kind in sorted(EDGES):
            with igr.Solver(_case(BIG, kind, solver, sweeps=1), "f16") as s:
                s.solve_sigma(q, s0.clone(), 1)
                s.sync()
    assert igr.lib().igr_debug_bounds_hits(C.byref(h), 1) == igr.OK and h.value == 0
    del s
    gc.collect()
