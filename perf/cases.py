"""The work this solver is used for, as timed cases.

A case is one pass of a user's program through the public entry points of
paper_2505_07392_gb300.igr and .adjoint, on inputs drawn on the GPU from a seed:

  step      set a state, advance SSP-RK3 steps, read the state (Solver)
  batch     the same for many independent instances together (Batch)
  adjoint   the discrete adjoint of one step (Solver.adjoint_step)
  autograd  one step and its gradients (adjoint.IGRStep)
  sigma     the elliptic solve alone (Solver.solve_sigma)
  rhs       the flux divergence alone (Solver.rhs)

exact() evaluates the same method in FP64 with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_2505_07392_gb300 import adjoint, igr, inputs

EDGES = (48, 64, 80, 96, 128)       # edges of the batched Taylor-Green boxes
EXACT_CELL_STEPS = 1.5e8            # exact() is worked out up to this many cell steps


def listed():
    def c(name, kind, flow, nx, ny, nz, precision, sweeps=5, steps=1, order=5, rbgs=False, mu=0.0, instances=1):
        return {"name": name, "kind": kind, "flow": flow, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
                "sweeps": sweeps, "steps": steps, "order": order, "rbgs": rbgs, "mu": mu, "instances": instances}

    return [
        # the benchmark's many-jet plume at a quarter of its height, in the headline storage form:
        # a production run's steps between two reads of the state
        c("plume_f16inc", "step", "plume", 1024, 1024, 512, "f16inc", steps=2),
        # the same flow on a parameter study's box in plain FP32
        c("plume_f32", "step", "plume", 512, 512, 256, "f32", steps=2),
        # the form that halves the memory: the whole state in FP16 (the box of the kernel profiles)
        c("plume_f16", "step", "plume", 512, 512, 128, "f16", steps=2),
        # Navier-Stokes with in-place red-black sweeps on a box whose edges fit no tile
        c("viscous_bf16inc_ragged", "step", "plume", 254, 201, 130, "bf16inc", steps=2, rbgs=True, mu=1e-4),
        # the spherical blast at its stated size and sweep count
        c("blast_f32", "step", "blast", 256, 256, 256, "f32", sweeps=10, steps=2),
        # the FP64 run that the other precisions are validated against
        c("blast_f64", "step", "blast", 96, 96, 96, "f64", sweeps=10, steps=2),
        # an ensemble of uneven Taylor-Green boxes advanced together
        c("batch_f16inc", "batch", "tgv", 0, 0, 0, "f16inc", steps=4, instances=16),
        # a unit-test-sized box: latency and launches
        c("wave_f32_32", "step", "wave", 32, 32, 32, "f32", steps=10),
        # the reverse sweep of the four-jet design problem, one step
        c("adjoint_f32", "adjoint", "jets4", 128, 128, 128, "f32"),
        # a differentiable step in a small FP64 optimisation loop, forward and backward
        c("autograd_f64_48", "autograd", "jets4", 48, 48, 48, "f64"),
        # the elliptic solve as an operator of its own
        c("sigma_f16", "sigma", "blast", 256, 256, 192, "f16", sweeps=5),
        # the spatial operator as a building block of another integrator, 3rd-order faces, odd edges
        c("rhs_f32_odd", "rhs", "tgv", 201, 119, 77, "f32", order=3),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "adjoint", "autograd", "sigma", "rhs"])
    hi = {"step": 2.6e8, "batch": 0, "adjoint": 4e6, "autograd": 1e6, "sigma": 1.2e8, "rhs": 6e7}[kind]
    case = {"kind": kind, "nx": 0, "ny": 0, "nz": 0, "order": 5, "rbgs": False, "mu": 0.0, "instances": 1,
            "sweeps": rng.choice([3, 5, 5, 5, 8, 10]), "steps": 1}
    if kind == "batch":
        case.update(flow="tgv", instances=rng.randint(4, 48), steps=rng.randint(2, 5), sweeps=5,
                    precision=rng.choice(["f16inc", "f32", "f16"]))
        return case
    case["flow"] = "jets4" if kind in ("adjoint", "autograd") else rng.choice(["plume", "plume", "blast", "tgv", "wave"])
    case["precision"] = rng.choice({"adjoint": ["f32", "f32", "f64"], "autograd": ["f32", "f64"]}.get(
        kind, ["f16inc", "f16inc", "f32", "f32", "f16", "bf16inc", "f64"]))
    if case["precision"] == "f64":
        hi = min(hi, 4e6)
    cells = math.exp(rng.uniform(math.log(2e4), math.log(hi)))
    # the box's shape; one time in two the edges are whole tiles or at least even, else whatever they come to
    ax, ay = math.exp(rng.uniform(-0.5, 0.5)), math.exp(rng.uniform(-0.5, 0.5))
    e = cells ** (1.0 / 3.0)
    dims = [e * ax, e * ay, e / (ax * ay)]
    unit = rng.choice([1, 1, 4, 32 if e > 100 else 2])
    case["nx"], case["ny"], case["nz"] = (max(8, int(round(d / unit)) * unit) for d in dims)
    if kind == "step":
        case["steps"] = max(1, min(10, int(2e8 / cells), rng.randint(1, 10)))
    if kind in ("step", "rhs"):
        case["order"] = rng.choice([5, 5, 5, 3])
        case["mu"] = rng.choice([0.0, 0.0, 0.0, 1e-4])
    if kind in ("step", "sigma") and case["flow"] in ("plume", "blast"):
        case["rbgs"] = rng.choice([False, False, False, True])
    return case


# ------------------------------------------------------------------ inputs

def _problems(case, seed):
    """The inputs.Case of every instance."""
    rng = np.random.Generator(np.random.Philox(seed))
    P, O, I = inputs.PERIODIC, inputs.OUTFLOW, inputs.INFLOW
    if case["kind"] == "batch":
        # the edges are the case's, the seed changes the flow alone
        pick = np.random.Generator(np.random.Philox(1000 + case["instances"])).choice(EDGES, size=case["instances"])
        boxes = [(int(e),) * 3 for e in pick]
    else:
        boxes = [(case["nx"], case["ny"], case["nz"])]
    made = []
    for nx, ny, nz in boxes:
        dx, jets, bc = 1.0 / nx, [], (P,) * 6
        if case["flow"] in ("plume", "jets4"):
            bc = (O, O, O, O, I, O)
            ref = inputs.plume(nx, ny, nz, seed=int(rng.integers(1 << 30))) if case["flow"] == "plume" else \
                inputs.jets4(nx)
            dx = ref.dx
            jets = [tuple(j[:4]) + (j[4] * float(1 + 0.02 * rng.uniform(-1, 1)),) + tuple(j[5:]) for j in ref.jets]
        elif case["flow"] == "blast":
            bc = (O,) * 6
        made.append(inputs.Case(case["flow"], nx, ny, nz, dx, alpha=dx * dx, sweeps=case["sweeps"], bc=bc, jets=jets,
                                order=case["order"], sigma_solver=int(case["rbgs"]), mu=case["mu"]))
    return made


def _state(p, seed, dtype):
    """The conserved state of problem p, built in slabs of planes: the flow's smooth fields, a large-scale
    velocity disturbance with phases from the seed, and density noise in every cell."""
    dev = "cuda"
    rng = np.random.Generator(np.random.Philox(seed + 7))
    ph = [float(v) for v in rng.uniform(0.0, 2 * math.pi, size=6)]
    gen = torch.Generator(device=dev).manual_seed(seed)
    q = torch.empty((5, p.nz, p.ny, p.nx), dtype=dtype, device=dev)
    f64 = torch.float64
    x = ((torch.arange(p.nx, dtype=f64, device=dev) + 0.5) / p.nx)[None, None, :]
    y = ((torch.arange(p.ny, dtype=f64, device=dev) + 0.5) / p.ny)[None, :, None]
    tau, g = 2 * math.pi, p.gamma
    if p.jets:
        W, J = _inflow(p)
        depth = 4.0 + 6.0 * float(rng.uniform())
    slab = max(1, int(3e7 // (p.nx * p.ny)))
    for k0 in range(0, p.nz, slab):
        k1 = min(p.nz, k0 + slab)
        kz = torch.arange(k0, k1, dtype=f64, device=dev)[:, None, None] + 0.5
        z = kz / p.nz
        noise = torch.rand((k1 - k0, p.ny, p.nx), generator=gen, dtype=torch.float32, device=dev) * 2 - 1
        du = 0.02 * torch.sin(tau * x + ph[0]) * torch.cos(tau * y + ph[1]) * torch.cos(tau * z + ph[2])
        dv = 0.02 * torch.cos(tau * x + ph[3]) * torch.sin(tau * y + ph[4]) * torch.cos(tau * z + ph[5])
        zero = torch.zeros_like(du)
        if p.name == "tgv":
            u = torch.sin(tau * x + ph[0]) * torch.cos(tau * y + ph[1]) * torch.cos(tau * z) + zero
            v = -torch.cos(tau * x + ph[0]) * torch.sin(tau * y + ph[1]) * torch.cos(tau * z) + zero
            w, rho, amp = zero, zero + 1.0, 0.05
            pr = 1.0 / (g * 0.25) + (torch.cos(2 * tau * x) + torch.cos(2 * tau * y)) * (torch.cos(2 * tau * z) + 2) / 16 + zero
        elif p.name == "wave":
            rho, amp = 1.0 + 0.2 * torch.sin(tau * x + ph[0]) + zero, 1e-3
            u, v, w, pr = 1.0 + du, dv, zero, zero + 1.0
        elif p.name == "blast":
            r = torch.sqrt(((x - 0.5) * p.nx) ** 2 + ((y - 0.5) * p.ny) ** 2 + ((z - 0.5) * p.nz) ** 2)
            s = 0.5 * (1.0 - torch.tanh(r - 0.2 * min(p.nx, p.ny, p.nz)))
            rho, pr, amp = 0.125 + 0.875 * s, 0.1 + 0.9 * s, 1e-4
            u, v, w = du, dv, zero
        else:  # a plug of jet gas at the inflow face in a gently stirred ambient
            f = 0.5 * (1.0 - torch.tanh(kz - depth))
            d = [f * (J[a] - W * a0)[None] for a, a0 in ((0, 1.0), (3, 0.0), (4, 1.0 / (g - 1.0)))]
            rho0, amp = 1.0 + d[0], 1e-3
            wz = d[1] / rho0
            pr = (g - 1.0) * (1.0 / (g - 1.0) + d[2] - 0.5 * rho0 * wz * wz)
            rho, u, v, w = rho0, du, dv, wz
        rho = rho * (1.0 + amp * noise.double())
        slot = q[:, k0:k1]
        slot[0], slot[1], slot[2], slot[3] = rho, rho * u, rho * v, rho * w
        slot[4] = pr / (g - 1.0) + 0.5 * rho * (u * u + v * v + w * w)
    return q


def _sigma(p, seed, dtype):
    """A warm start: Sigma of the size alpha |grad u|^2 has where the flow is compressed."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 31)
    s = torch.rand((p.nz, p.ny, p.nx), generator=gen, dtype=torch.float32, device="cuda")
    return (0.01 * s).to(dtype)


def _weights(p, seed, dtype):
    """Adjoints of a step's results, of the size a mean over the box gives them."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 57)
    n = (6, p.nz, p.ny, p.nx)
    w = torch.rand(n, generator=gen, dtype=torch.float32, device="cuda") * 2 - 1
    return w[:5].to(dtype).contiguous(), w[5].to(dtype).contiguous()


FIXED_DT = 0.2  # of a cell per unit speed: the frozen step of the differentiated cases


def prepare(case, seed):
    probs = _problems(case, seed)
    prec, kind = case["precision"], case["kind"]
    qt, st, ct = igr.state_torch_dtype(prec), igr.storage_torch_dtype(prec), igr.compute_torch_dtype(prec)
    if kind == "batch":
        return {"case": case, "batch": igr.Batch(probs, prec), "q": [_state(p, seed + 97 * i, qt) for i, p in enumerate(probs)]}
    p = probs[0]
    s = {"case": case, "solver": igr.Solver(p, prec), "q": _state(p, seed, qt)}
    if kind != "step":
        s["sigma"] = _sigma(p, seed, st)
    if kind in ("adjoint", "autograd"):
        s["lam_q"], s["lam_sigma"] = _weights(p, seed, ct)
        s["dt"] = FIXED_DT * p.dx
    if kind == "autograd":
        s["q"], s["sigma"] = s["q"].to(ct).requires_grad_(True), s["sigma"].to(ct).requires_grad_(True)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "step":
        sol = s["solver"]
        sol.set_state(s["q"])
        sol.step(case["steps"], sync=False)
        q, sigma = sol.get_state()
        # Sigma is kept in its storage type (exact)
        return {"q": q, "sigma": sigma.to(igr.storage_torch_dtype(case["precision"]))}
    if kind == "batch":
        b = s["batch"]
        for inst, q in zip(b.instances, s["q"]):
            inst.set_state(q)
        b.step(case["steps"])
        b.sync()
        return [inst.get_state()[0] for inst in b.instances]
    if kind == "adjoint":
        lq, ls, gw = s["solver"].adjoint_step(s["q"], s["sigma"], s["lam_q"], s["lam_sigma"], s["dt"])
        return {"lam_q": lq, "lam_sigma": ls, "jets": np.array(gw)}
    if kind == "autograd":
        q1, s1 = adjoint.IGRStep.apply(s["q"], s["sigma"], s["solver"], s["dt"])
        gq, gs = torch.autograd.grad((q1, s1), (s["q"], s["sigma"]), (s["lam_q"], s["lam_sigma"]))
        return {"q": q1.detach(), "sigma": s1.detach(), "lam_q": gq, "lam_sigma": gs}
    if kind == "sigma":
        return s["solver"].solve_sigma(s["q"], s["sigma"].clone(), case["sweeps"])
    return s["solver"].rhs(s["q"], s["sigma"])


def work(case):
    """A step reads the state and Sigma once and writes them once (its dt needs a maximum over the whole state,
    so every step does); a face's reconstruction is 108 operations, its flux about 70, a sweep 27, the source 45."""
    prec, kind = case["precision"], case["kind"]
    size = {"f64": (8, 8), "f32": (4, 4), "f16": (2, 2), "bf16": (2, 2), "f16inc": (4, 2), "bf16inc": (4, 2)}
    qb, sb = size[prec]
    cb = 8 if prec == "f64" else 4
    n = sum(p.ncells for p in _problems(case, 0))
    flux, sweep, source = 3 * 178 + 60, 27 * case["sweeps"], 45
    step = 3 * (flux + sweep + source)
    if kind in ("step", "batch"):
        return {"bytes": n * case["steps"] * 2 * (5 * qb + sb), "flops": n * case["steps"] * step}
    if kind == "adjoint":
        return {"bytes": n * (5 * qb + sb + 12 * cb), "flops": 3 * n * step}
    if kind == "autograd":
        return {"bytes": n * (5 * qb + sb + 18 * cb), "flops": 4 * n * step}
    if kind == "sigma":
        return {"bytes": n * (4 * qb + 2 * sb), "flops": n * (sweep + source)}
    return {"bytes": n * (5 * qb + sb + 5 * cb), "flops": n * flux}


# ------------------------------------------------- the method in FP64 torch

def _inflow(p):
    """Blend weight W and weighted jet state J of the -z face, (ny, nx) and (5, ny, nx)."""
    f64 = torch.float64
    x = ((torch.arange(p.nx, dtype=f64, device="cuda") + 0.5) * p.dx)[None, :]
    y = ((torch.arange(p.ny, dtype=f64, device="cuda") + 0.5) * p.dx)[:, None]
    W = torch.zeros((p.ny, p.nx), dtype=f64, device="cuda")
    J = torch.zeros((5, p.ny, p.nx), dtype=f64, device="cuda")
    for cx, cy, R, rho, w, pr, edge in p.jets:
        s = 0.5 * (1.0 - torch.tanh((torch.sqrt((x - cx) ** 2 + (y - cy) ** 2) - R) / (edge * p.dx)))
        W += s
        J[0] += s * rho
        J[3] += s * rho * w
        J[4] += s * (pr / (p.gamma - 1.0) + 0.5 * rho * w * w)
    return W, J


def _grow(f, axis, h, periodic):
    """f with h more cells on both sides of axis (0 z, 1 y, 2 x; the last three dimensions): wrapped or copied."""
    d = f.dim() - 3 + axis
    n = f.shape[d]
    at = torch.arange(-h, n + h, device=f.device)
    return f.index_select(d, at % n if periodic else at.clamp(0, n - 1))


class _Exact:
    def __init__(self, p):
        self.p, self.W, self.J = p, *_inflow(p)
        self.per = [p.bc[4] == 0, p.bc[2] == 0, p.bc[0] == 0]  # of the axes z, y, x

    def grow(self, f, axis, h, W=None, J=None):
        """As _grow; fields f (first dimension) that a jet face blends get its ghosts below z."""
        e = _grow(f, axis, h, self.per[axis])
        if axis == 0 and self.p.bc[4] == inputs.INFLOW and J is not None:
            ghost = (1.0 - W) * e[:, :h] + J[:, None]
            e = torch.cat([ghost, e[:, h:]], 1)
        return e

    def cut(self, f, axis, a, b):
        d = f.dim() - 3 + axis
        return f.narrow(d, a, b - a)

    def source(self, q):
        p = self.p
        G = {}
        for axis, c in ((2, 0), (1, 1), (0, 2)):
            e = self.grow(q[:4], axis, 1, self.W, self.J[:4])
            u = e[1:] / e[0]
            n = q.shape[1 + axis]
            d = (self.cut(u, axis, 2, n + 2) - self.cut(u, axis, 0, n)) / (2 * p.dx)
            for a in range(3):
                G[a, c] = d[a]
        tr = G[0, 0] + G[1, 1] + G[2, 2]
        t2 = sum(G[a, c] * G[c, a] for a in range(3) for c in range(3))
        return p.alpha * (t2 + tr * tr)

    def sweeps(self, rho, b, s, count):
        p = self.p
        beta, r = p.alpha / (p.dx * p.dx), 1.0 / rho
        diag, faces = r, []
        for axis in range(3):
            n = r.shape[axis]
            er = _grow(r, axis, 1, self.per[axis])
            for side in (0, 2):
                c = 0.5 * beta * (r + self.cut(er, axis, side, side + n))
                if not self.per[axis]:  # no term across the boundary
                    keep = torch.ones(n, dtype=r.dtype, device=r.device)
                    keep[0 if side == 0 else n - 1] = 0.0
                    c = c * keep.reshape([n if a == axis else 1 for a in range(3)])
                diag = diag + c
                faces.append((axis, side, n, c))

        def update(s):
            off = b
            for axis in range(3):
                es = _grow(s, axis, 1, self.per[axis])
                for ax, side, n, c in faces:
                    if ax == axis:
                        off = off + c * self.cut(es, axis, side, side + n)
            return off / diag

        if not p.sigma_solver:
            for _ in range(count):
                s = update(s)
            return s
        k, j, i = (torch.arange(n, device=r.device) for n in r.shape)
        red = ((i[None, None, :] + j[None, :, None] + k[:, None, None]) % 2) == 0
        for _ in range(count):
            s = torch.where(red, update(s), s)
            s = torch.where(red, s, update(s))
        return s

    def physical(self, v, D):
        p = self.p
        rho, m, E, sig = v[0], v[1:4], v[4], v[5]
        u = m[D] / rho
        pr = (p.gamma - 1.0) * (E - 0.5 * (m * m).sum(0) / rho)
        F = [m[D]] + [m[a] * u + (pr + sig if a == D else 0.0) for a in range(3)] + [(E + pr + sig) * u]
        return F, u.abs() + torch.sqrt(p.gamma * pr / rho)

    def viscous(self, q, axis, D):
        """Viscous flux through every face across `axis`: momentum along each direction, energy."""
        p = self.p
        W, J = _grow(_grow(self.W[None, None], 1, 1, self.per[1]), 2, 1, self.per[2])[0, 0], \
            _grow(_grow(self.J[:, None], 1, 1, self.per[1]), 2, 1, self.per[2])[:, 0]
        e = self.grow(self.grow(q[:4], 2, 1), 1, 1)
        e = self.grow(e, 0, 1, W, J[:4])
        u = e[1:] / e[0]  # one cell more on every side
        dim = {0: 2, 1: 1, 2: 0}  # the axis of each direction
        n = [q.shape[1 + a] for a in range(3)]

        def at(f, shift):  # cells -1..n along `axis` (n + 2 of them) and the own ones elsewhere, shifted
            for a in range(3):
                sh = shift.get(a, 0)
                f = f if a == axis else self.cut(f, a, 1 + sh, n[a] + 1 + sh)
            return f

        lo = lambda f: self.cut(f, axis, 0, n[axis] + 1)  # noqa: E731
        up = lambda f: self.cut(f, axis, 1, n[axis] + 2)  # noqa: E731
        c = at(u, {})
        g = {}
        for d in range(3):
            a = dim[d]
            if a == axis:
                g[d] = (up(c) - lo(c)) / p.dx
            else:
                t = (at(u, {a: 1}) - at(u, {a: -1})) / (2 * p.dx)
                g[d] = 0.5 * (lo(t) + up(t))
        div = g[0][0] + g[1][1] + g[2][2]
        tau = [p.mu * (g[D][a] + g[a][D]) + ((p.zeta - 2 * p.mu / 3) * div if a == D else 0.0) for a in range(3)]
        uf = 0.5 * (lo(c) + up(c))
        return tau, sum(uf[a] * tau[a] for a in range(3))

    def rhs(self, q, sig):
        p = self.p
        out = torch.zeros_like(q)
        if p.order == 3:
            wl, wr = (0, -1 / 6, 5 / 6, 2 / 6, 0, 0), (0, 0, 2 / 6, 5 / 6, -1 / 6, 0)
        else:
            wl, wr = (2 / 60, -13 / 60, 47 / 60, 27 / 60, -3 / 60, 0), (0, -3 / 60, 27 / 60, 47 / 60, -13 / 60, 2 / 60)
        for axis, D in ((2, 0), (1, 1), (0, 2)):
            n = q.shape[1 + axis]
            e = torch.cat([self.grow(q, axis, 3, self.W, self.J), _grow(sig[None], axis, 3, self.per[axis])])
            pts = [self.cut(e, axis, m, m + n + 1) for m in range(6)]
            L = sum(w * v for w, v in zip(wl, pts) if w)
            R = sum(w * v for w, v in zip(wr, pts) if w)
            FL, aL = self.physical(L, D)
            FR, aR = self.physical(R, D)
            lam = torch.where(aL > aR, aL, aR)
            F = [0.5 * (FL[v] + FR[v] - lam * (R[v] - L[v])) for v in range(5)]
            if p.mu or p.zeta:
                tau, heat = self.viscous(q, axis, D)
                F = [F[0]] + [F[1 + a] - tau[a] for a in range(3)] + [F[4] - heat]
            out = out - torch.stack([self.cut(f, axis, 1, n + 1) - self.cut(f, axis, 0, n) for f in F]) / p.dx
        return out

    def step(self, q, s, dt=None):
        p = self.p
        if dt is None:
            m = q[1:4].abs().amax(0) / q[0]
            pr = (p.gamma - 1.0) * (q[4] - 0.5 * (q[1:4] ** 2).sum(0) / q[0])
            dt = float(p.cfl * p.dx / (m + torch.sqrt(p.gamma * pr / q[0])).max())
        qs = q
        for w in (1.0, 0.25, 2.0 / 3.0):
            s = self.sweeps(qs[0], self.source(qs), s, p.sweeps)
            qs = q + w * ((qs - q) + dt * self.rhs(qs, s))
        return qs, s


def exact(case, seed):
    probs = _problems(case, seed)
    if sum(p.ncells for p in probs) * case["steps"] > EXACT_CELL_STEPS:
        return None
    prec, kind = case["precision"], case["kind"]
    qt, st, ct = igr.state_torch_dtype(prec), igr.storage_torch_dtype(prec), igr.compute_torch_dtype(prec)
    f64 = torch.float64
    if kind in ("step", "batch"):
        done = []
        for i, p in enumerate(probs):
            q, e = _state(p, seed + 97 * i, qt).to(f64), _Exact(p)
            s = torch.zeros_like(q[0])
            for _ in range(case["steps"]):
                q, s = e.step(q, s)
            done.append((q, s))
        return [q for q, _ in done] if kind == "batch" else {"q": done[0][0], "sigma": done[0][1]}
    p = probs[0]
    e = _Exact(p)
    q, s = _state(p, seed, qt).to(f64), _sigma(p, seed, st).to(f64)
    if kind == "sigma":
        return e.sweeps(q[0], e.source(q), s, case["sweeps"])
    if kind == "rhs":
        return e.rhs(q, s)
    lq, ls = (w.to(f64) for w in _weights(p, seed, ct))
    q.requires_grad_(True)
    s.requires_grad_(True)
    J = e.J
    jw = torch.tensor([j[4] for j in p.jets], dtype=f64, device="cuda", requires_grad=True)
    e.J = _jets_of(p, J, jw)
    q1, s1 = e.step(q, s, FIXED_DT * p.dx)
    gq, gs, gw = torch.autograd.grad((q1, s1), (q, s, jw), (lq, ls))
    if kind == "adjoint":
        return {"lam_q": gq, "lam_sigma": gs, "jets": gw}
    return {"q": q1.detach(), "sigma": s1.detach(), "lam_q": gq, "lam_sigma": gs}


def _jets_of(p, J, jw):
    """The weighted jet state as a function of the jets' velocities jw."""
    f64 = torch.float64
    x = ((torch.arange(p.nx, dtype=f64, device="cuda") + 0.5) * p.dx)[None, :]
    y = ((torch.arange(p.ny, dtype=f64, device="cuda") + 0.5) * p.dx)[:, None]
    mz, E = torch.zeros_like(J[3]), torch.zeros_like(J[4])
    for k, (cx, cy, R, rho, _, pr, edge) in enumerate(p.jets):
        s = 0.5 * (1.0 - torch.tanh((torch.sqrt((x - cx) ** 2 + (y - cy) ** 2) - R) / (edge * p.dx)))
        mz = mz + s * rho * jw[k]
        E = E + s * (pr / (p.gamma - 1.0) + 0.5 * rho * jw[k] ** 2)
    return torch.stack([J[0], J[1], J[2], mz, E])
