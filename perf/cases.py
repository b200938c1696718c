"""Performance cases of libgpeshell: what a user's program has the library do,
each as one pass through the public calls of ``paper_2603_05447_gb300.gpe``
and ``.autograd``.

A case is a dict of plain values.  ``kind`` says which calls a pass makes:

* ``real``   RK steps in real time (traced every ``every`` steps if that is
             not 0), then the state stored to the caller's array;
* ``imag``   imaginary-time steps, the observables (one check block of a
             ground-state solve), then the state stored;
* ``batch``  a check block of a batch of uneven shells from fresh states;
* ``grad``   loss and knot gradient of a ramp through torch.autograd;
* ``stages`` a multi-stage ramp over dense potentials, regridding per stage.

Geometries: ``trap`` (isotropic harmonic trap, every cell active), ``shell``
(thin ellipsoidal shell, V < 5 mu0 active) and ``ramp`` (harmonic core blended
into a shell, both regions active), with the closed forms of the workloads in
``inputs.py``.  Initial states are Thomas-Fermi-like profiles (a Gaussian in
the trap) with seeded noise.
"""
import gc
import math

import numpy as np
import torch

from paper_2603_05447_gb300 import gpe
from paper_2603_05447_gb300.autograd import RampProblem, ramp_infidelity

DTYPES = {"c128": (gpe.GPE_C128, torch.complex128), "c64": (gpe.GPE_C64, torch.complex64),
          "r64": (gpe.GPE_R64, torch.float64), "r32": (gpe.GPE_R32, torch.float32)}
INTEGRATORS = {"rk4": gpe.GPE_RK4, "rkhe3": gpe.GPE_RKHE3, "rkck": gpe.GPE_RKCK}
OBS = ("norm", "energy", "mu", "e_kin", "e_pot", "e_int")
DEV = "cuda"
N_ATOMS = 1.0

_side = None


def _stream():
    """One non-default stream for every state, as a program keeps one (the
    library replays step loops as CUDA graphs there)."""
    global _side
    if _side is None:
        _side = torch.cuda.Stream()
    return _side


# ------------------------------------------------------------------ the cases
def _case(kind, geometry, **kw):
    c = dict(kind=kind, geometry=geometry, dtype="c64", brick="8x8x4", stencil=7, integrator="rk4", g=2000.0,
             a_cells=0.0, ab=0.9, ac=0.8, width=6.0, sy=1.0, sz=1.0, n=0, steps=1, every=0, shells=0, stages=0)
    c.update(kw)
    return c


def listed():
    return [
        # a program that steps a small trap one step at a time (own control loop): launches and latency
        _case("real", "trap", name="trap64 single RK4 step c64", n=64, g=100.0, brick="8x8x8", steps=1),
        # the harmonic-trap ground-state run in FP64: one check block of 50 steps
        _case("imag", "trap", name="trap64 ground state c128", n=64, g=100.0, dtype="c128", brick="8x8x8", steps=50),
        # the headline: real-time evolution of the 1024^3 shell in complex64
        _case("real", "shell", name="shell1024 RK4 c64", n=1024, a_cells=490.0, steps=32),
        # the same evolution in full precision (the accuracy reference of the runs above)
        _case("real", "shell", name="shell1024 RK4 c128", n=1024, a_cells=490.0, dtype="c128", steps=4),
        # the other integrators, default bricks, half-size shell
        _case("real", "shell", name="shell512 RKCK c64", n=512, a_cells=240.0, brick="8x8x8",
              integrator="rkck", steps=8),
        # higher-order stencil
        _case("real", "shell", name="shell1024 RK4 19-point c64", n=1024, a_cells=490.0, stencil=19, steps=8),
        # ground state of the headline shell: a check block of 10 steps and its observables
        _case("imag", "shell", name="shell1024 ground state c64", n=1024, a_cells=490.0, steps=10),
        # real-valued ground state, default bricks
        _case("imag", "shell", name="shell512 ground state r32", n=512, a_cells=240.0, dtype="r32",
              brick="8x8x8", steps=10),
        # the tracked hollowing-out ramp at full size
        _case("real", "ramp", name="ramp2048 traced c64", n=2048, a_cells=800.0, g=5000.0,
              brick="8x8x8", steps=12, every=4),
        # many uneven shells in one launch
        _case("batch", "shell", name="batch of 8 shells c64", a_cells=360.0, brick="8x8x8", shells=8, steps=20),
        # gradient of the ramp infidelity with respect to the 16 knots
        _case("grad", "ramp", name="ramp512 gradient c64", n=512, a_cells=200.0, g=5000.0, brick="8x8x8", steps=48),
        # precomputed dense potentials: Thomas-Fermi solves, regrids, remaps and steps
        _case("stages", "shell", name="stages512 dense f32", n=512, a_cells=240.0, stages=4, steps=20),
    ]


def draw(rng):
    def loguniform(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["real"] * 5 + ["imag"] * 4 + ["batch", "grad", "stages"])
    brick = rng.choice(["8x8x8", "8x8x8", "8x8x4", "8x4x4"])
    shape = dict(ab=round(rng.uniform(0.7, 1.0), 3), ac=round(rng.uniform(0.7, 1.0), 3),
                 width=round(rng.uniform(4.0, 10.0), 2), sy=round(rng.uniform(0.95, 1.1), 3),
                 sz=round(rng.uniform(0.95, 1.1), 3), g=round(loguniform(100.0, 5000.0), 1), brick=brick)
    if kind == "grad":
        c = _case("grad", "ramp", a_cells=round(loguniform(20.0, 200.0), 1), steps=rng.randint(9, 48), **shape)
        c["dtype"] = rng.choice(["c64", "c64", "c128"]) if c["a_cells"] < 100 else "c64"
        return c
    if kind == "stages":
        return _case("stages", "shell", a_cells=round(loguniform(30.0, 240.0), 1), stages=rng.randint(2, 4),
                     steps=rng.randint(5, 20), **shape)
    if kind == "batch":
        return _case("batch", "shell", a_cells=round(loguniform(40.0, 300.0), 1), shells=rng.randint(3, 12),
                     steps=rng.randint(5, 20), dtype=rng.choice(["c64", "r32"]), **shape)
    if rng.random() < 0.25:
        c = _case(kind, "trap", **dict(shape, n=rng.randint(24, 96), g=round(loguniform(1.0, 300.0), 2)))
    elif kind == "real" and rng.random() < 0.3:
        c = _case(kind, "ramp", a_cells=round(loguniform(20.0, 400.0), 1), **shape)
    else:
        c = _case(kind, "shell", a_cells=round(loguniform(20.0, 480.0), 1), **shape)
    c["dtype"] = rng.choice(["c64", "c64", "c128"] if kind == "real" else ["c64", "c64", "r32", "c128", "r64"])
    if rng.random() < 0.2:
        c["stencil"] = 19
    elif kind == "real" and rng.random() < 0.3:
        c["integrator"] = rng.choice(["rkhe3", "rkck"])
    w = work(dict(c, steps=1))
    most_flops = 8e11 if c["dtype"] in ("c128", "r64") else 4e12
    most = max(1, min(40, int(min(2e10 / w["bytes"], most_flops / w["flops"]))))
    c["steps"] = rng.randint(1, most)
    if kind == "real" and c["steps"] > 1 and rng.random() < 0.3:
        c["every"] = rng.randint(1, c["steps"])
    return c


# ------------------------------------------------------------------ the problem in numbers
class _Problem:
    """Box, potentials, cutoffs and time steps of one grid of a case."""

    def __init__(self, case):
        self.g = case["g"]
        self.brick = tuple(int(v) for v in case["brick"].split("x"))
        sy, sz = case["sy"], case["sz"]
        if case["geometry"] == "trap":
            n = case["n"]
            h = 16.0 / n
            self.dims = (n, max(8, round(n / sy)), max(8, round(n / sz)))
            self.spacing = (h, h * sy, h * sz)
            self.pots = [("harmonic", (1.0, 1.0, 1.0), math.inf)]
            vmax = 0.5 * sum((0.5 * (m - 1) * s) ** 2 for m, s in zip(self.dims, self.spacing))
            self.mu0 = 0.5 * (15.0 * self.g * N_ATOMS / (4.0 * math.pi)) ** 0.4
            self.n_active = math.prod(self.dims)
            self.dt_imag = 1e-3
        else:
            ac = case["a_cells"]
            axes = (1.0, case["ab"], case["ac"])
            u = 0.5 * case["width"] / ac
            band = math.sqrt(5.0) * u
            mu0 = 3.0 * self.g * N_ATOMS / (16.0 * math.pi * axes[1] * axes[2] * u)
            w = math.sqrt(2.0 * mu0) / u
            h = 1.0 / ac
            self.spacing = (h, h * sy, h * sz)
            # a cubic box of n cells, or (n = 0) the band's own box with a margin, odd unless the spacings are equal
            self.dims = (case["n"],) * 3 if case["n"] else tuple(
                int(2 * math.ceil(a * (1.0 + band) / s + 4)) + (1 if sy != 1.0 else 0)
                for a, s in zip(axes, self.spacing))
            shell = ("shell", (w,) + axes, 5.0 * mu0)
            vol = 4.0 / 3.0 * math.pi * axes[1] * axes[2] * ((1.0 + band) ** 3 - max(0.0, 1.0 - band) ** 3)
            vmax = 5.0 * mu0
            self.mu0 = mu0
            self.pots = [shell]
            if case["geometry"] == "ramp":
                core = 0.24
                r = core / math.sqrt(5.0)
                c = (15.0 * self.g * N_ATOMS / (4.0 * math.pi)) ** 0.4
                wc = (c / r ** 2) ** (1.0 / 0.8)
                self.mu0 = 0.5 * wc * wc * r * r
                self.pots = [("harmonic", (wc, wc, wc), 5.0 * self.mu0), shell]
                vol += 4.0 / 3.0 * math.pi * core ** 3
                # either potential over both regions (the blend's largest value on active cells)
                vmax = max(0.5 * wc * wc * (1.0 + band) ** 2, 0.5 * w * w, 5.0 * self.mu0)
            self.n_active = int(vol / math.prod(self.spacing))
            self.dt_imag = min(0.5 * min(self.spacing) ** 2, 0.5 / mu0)
        kin = sum(2.0 / s ** 2 for s in self.spacing)
        self.dt_real = 0.2 / (kin + vmax + 2.0 * self.mu0)
        self.dV = math.prod(self.spacing)
        self.origin = tuple(-(m - 1) / 2.0 * s for m, s in zip(self.dims, self.spacing))

    def box(self):
        return gpe.make_box(*self.dims, *self.spacing, *self.origin)

    def grid(self, stencil=7):
        opts = gpe.make_opts(self.brick, stencil=stencil)
        kinds = {"harmonic": gpe.GPE_POT_HARMONIC, "shell": gpe.GPE_POT_ELLIPSOID_SHELL}
        pots = [(gpe.make_potential(kinds[k], *p), cut) for k, p, cut in self.pots]
        if len(pots) == 2:
            return gpe.gpe_grid_create_blend(self.box(), *pots[0], *pots[1], opts)
        return gpe.gpe_grid_create_analytic(self.box(), *pots[0], opts)


def _shells(case):
    """The shells of a batch: uneven radii, aspects, thicknesses and couplings."""
    import random
    rng = random.Random(4)
    return [_Problem(dict(case, a_cells=case["a_cells"] * rng.uniform(0.5, 1.0), ab=rng.uniform(0.7, 1.0),
                          ac=rng.uniform(0.7, 1.0), width=rng.uniform(4.0, 10.0), g=rng.uniform(100.0, 3000.0)))
            for _ in range(case["shells"])]


def _knots(seed):
    inner = np.sort(np.random.default_rng(seed).uniform(0.0, 1.0, 14))
    return np.concatenate([[0.0], inner, [1.0]]).tolist()


def _initial(P, V, case, seed, dtype):
    """The initial state on cells with potential V (+inf: inactive), normalised."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    a = torch.randn(V.numel(), generator=gen, device=DEV, dtype=torch.float64)
    if case["geometry"] == "trap":
        b = torch.randn(V.numel(), generator=gen, device=DEV, dtype=torch.float64)
        psi = torch.exp(-V) + (1e-3 * torch.complex(a, b) if dtype.is_complex else 1e-3 * a)
        psi = torch.where(torch.isinf(V), torch.zeros_like(psi), psi)
    else:
        amp = torch.sqrt(torch.clamp(P.mu0 - V, min=0.0) / P.g)
        psi = torch.polar(amp, 0.1 * a) if dtype.is_complex else amp * (1.0 + 0.01 * a)
    psi *= math.sqrt(N_ATOMS / (psi.abs().square().sum().item() * P.dV))
    return psi.to(dtype)


# ------------------------------------------------------------------ states
class _State:
    """What a program keeps: handles (destroyed with it) and device arrays."""

    def __init__(self, case, P):
        self.case, self.P = case, P
        self.grids, self.states, self.others = [], [], []

    def add(self, P, seed, case, dtype):
        grid = P.grid(case["stencil"])
        self.grids.append(grid)
        st = gpe.gpe_state_create(grid, DTYPES[dtype][0])
        self.states.append(st)
        V = torch.from_numpy(gpe.gpe_grid_potential(grid, 0)).to(DEV)
        return grid, st, _initial(P, V, case, seed, DTYPES[dtype][1])

    def __del__(self):
        torch.cuda.synchronize()
        for f, h in self.others:
            f(h)
        for s in self.states:
            gpe.gpe_state_destroy(s)
        for g in self.grids:
            gpe.gpe_grid_destroy(g)


def prepare(case, seed):
    gc.collect()
    S = _State(case, _Problem(case))
    with torch.cuda.stream(_stream()):
        {"real": _prepare_one, "imag": _prepare_one, "batch": _prepare_batch, "grad": _prepare_grad,
         "stages": _prepare_stages}[case["kind"]](S, case, seed)
    torch.cuda.synchronize()
    return S


def _prepare_one(S, case, seed):
    P = S.P
    _, S.st, psi = S.add(P, seed, case, case["dtype"])
    gpe.gpe_state_load(S.st, psi, gpe.GPE_LAYOUT_COMPACT)
    S.out = torch.empty_like(psi)
    if case["kind"] == "imag":
        S.params = gpe.gpe_imag_params(P.g, P.dt_imag, N_ATOMS)
    elif case["geometry"] == "ramp":
        S.params = gpe.real_params(P.g, P.dt_real, gpe.GPE_V_BLEND, _knots(seed), case["steps"] * P.dt_real,
                                   INTEGRATORS[case["integrator"]])
    else:
        S.params = gpe.real_params(P.g, P.dt_real, integrator=INTEGRATORS[case["integrator"]])


def _prepare_batch(S, case, seed):
    S.psi = [S.add(P, seed * 100 + i, case, case["dtype"])[2] for i, P in enumerate(_shells(case))]
    S.out = [torch.empty_like(p) for p in S.psi]
    S.params = [gpe.gpe_imag_params(P.g, P.dt_imag, N_ATOMS) for P in _shells(case)]
    S.batch = gpe.gpe_batch_create(S.states)
    S.others.append((gpe.gpe_batch_destroy, S.batch))


def _prepare_grad(S, case, seed):
    P = S.P
    grid, _, psi = S.add(P, seed, case, case["dtype"])
    V = torch.from_numpy(gpe.gpe_grid_potential(grid, 0)).to(DEV)
    target = _initial(P, V, case, seed + 1, DTYPES[case["dtype"]][1])
    # checkpoints every third of the run
    S.problem = RampProblem(grid, DTYPES[case["dtype"]][0], psi, target, P.g, P.dt_real, case["steps"],
                            case["steps"] * P.dt_real, K=max(1, case["steps"] // 3))
    S.others.append((RampProblem.close, S.problem))
    S.knots = torch.tensor(_knots(seed), dtype=torch.float32, requires_grad=True)


def _stage_potentials(case, P):
    """Dense FP32 potentials: even blends of the shell and a softer, rounder one."""
    (_, (w, a, b, c), _), = P.pots
    x, y, z = (o + torch.arange(n, dtype=torch.float64, device=DEV) * s
               for n, s, o in zip(P.dims, P.spacing, P.origin))

    def shell(w, a, b, c):
        rho = torch.sqrt((x / a).square() + (y / b).square()[:, None] + (z / c).square()[:, None, None])
        return 0.5 * w * w * (rho - 1.0).square()

    V0, V1 = shell(w, a, b, c), shell(0.6 * w, a, b + 0.01, c + 0.02)
    n = case["stages"]
    return [torch.lerp(V0, V1, k / n).to(torch.float32).contiguous() for k in range(n + 1)]


def _prepare_stages(S, case, seed):
    P = S.P
    S.pots = _stage_potentials(case, P)
    grid = gpe.gpe_grid_create_dense(P.box(), S.pots[0], P.pots[0][2], gpe.make_opts(P.brick))
    S.grids.append(grid)
    S.st = gpe.gpe_state_create(grid, DTYPES[case["dtype"]][0])
    S.states.append(S.st)
    V = torch.from_numpy(gpe.gpe_grid_potential(grid, 0)).to(DEV)
    gpe.gpe_state_load(S.st, _initial(P, V, case, seed, DTYPES[case["dtype"]][1]), gpe.GPE_LAYOUT_COMPACT)
    dt = 0.5 * P.dt_real  # a stage's region reaches beyond V < 5 mu0 of the first potential
    S.durations = [case["steps"] * dt] * case["stages"]
    S.params = gpe.stage_params(P.g, N_ATOMS, dt)


# ------------------------------------------------------------------ one pass
def run(S):
    case = S.case
    with torch.cuda.stream(_stream()):
        if case["kind"] == "real":
            if case["every"]:
                trace = gpe.gpe_step_real_traced(S.st, S.params, case["steps"], case["every"])
                gpe.gpe_state_store(S.st, S.out, gpe.GPE_LAYOUT_COMPACT)
                return {"psi": S.out, "trace": [[o[k] for k in OBS] for o in trace]}
            gpe.gpe_step_real(S.st, S.params, case["steps"])
            gpe.gpe_state_store(S.st, S.out, gpe.GPE_LAYOUT_COMPACT)
            return {"psi": S.out}
        if case["kind"] == "imag":
            gpe.gpe_step_imag(S.st, S.params, case["steps"])
            o = gpe.gpe_observables(S.st, S.P.g)
            gpe.gpe_state_store(S.st, S.out, gpe.GPE_LAYOUT_COMPACT)
            return {"psi": S.out, "obs": [o[k] for k in OBS]}
        if case["kind"] == "batch":
            for st, psi in zip(S.states, S.psi):
                gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_COMPACT)
            _, _, _, obs = gpe.gpe_batch_ground_state(S.batch, S.params, 1e-8, case["steps"], case["steps"],
                                                      check=False)
            for st, out in zip(S.states, S.out):
                gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_COMPACT)
            return {"psi": S.out, "obs": [[o[k] for k in OBS] for o in obs]}
        if case["kind"] == "grad":
            S.knots.grad = None
            loss = ramp_infidelity(S.knots, S.problem)
            loss.backward()
            out = torch.empty(gpe.gpe_grid_get_info(S.grids[0]).n_packed, dtype=DTYPES[case["dtype"]][1], device=DEV)
            gpe.gpe_state_store(S.problem.state, out, gpe.GPE_LAYOUT_COMPACT)
            return {"loss": loss.item(), "grad": S.knots.grad, "psi": out}
        grid, st, rep = gpe.gpe_ramp_stages(S.st, S.pots, S.durations, S.params)
        out = torch.empty(gpe.gpe_grid_get_info(grid).n_packed, dtype=DTYPES[case["dtype"]][1], device=DEV)
        gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_COMPACT)
        gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(grid)
        return {"psi": out, "n_active": [r["n_active"] for r in rep],
                "report": [[r[k] for k in ("mu_a", "mu_b", "cut", "norm_kept", "norm_end")] for r in rep]}


# ------------------------------------------------------------------ bytes and operations
def work(case):
    """Per active cell and step: psi in and out, every potential in (the table
    exp(-V dt/2) in imaginary time); 7-point Laplacian and update per stage."""
    size = {"c64": (8, 4), "c128": (16, 8), "r32": (4, 4), "r64": (8, 8)}[case["dtype"]]
    parts = 2 if case["dtype"].startswith("c") else 1
    per_stage = (38 if case["stencil"] == 7 else 82) * parts / 2 * (1 if parts == 2 else 1.1)
    if case["kind"] == "batch":
        cells = sum(P.n_active for P in _shells(case))
    else:
        cells = _Problem(case).n_active
    steps = case["steps"]
    if case["kind"] in ("imag", "batch"):
        # a step is two stencil passes; one more pass for the observables
        return {"bytes": cells * ((2 * size[0] + size[1]) * steps + size[0] + size[1]),
                "flops": cells * per_stage * (2 * steps + 1)}
    n_stage = {"rk4": 4, "rkhe3": 3, "rkck": 6}[case["integrator"]]
    pots = 2 if case["geometry"] == "ramp" or case["kind"] == "stages" else 1
    step_bytes, step_flops = 2 * size[0] + pots * size[1], n_stage * per_stage
    if case["kind"] == "grad":
        # forward, the recomputed states, and the reverse step (state, adjoint in and out)
        return {"bytes": cells * steps * (2 * step_bytes + 3 * size[0] + 2 * size[1]),
                "flops": cells * steps * step_flops * 4}
    if case["kind"] == "stages":
        dense = 4 * math.prod(_Problem(case).dims)
        return {"bytes": case["stages"] * (cells * step_bytes * steps + 2 * dense) + (case["stages"] + 1) * dense,
                "flops": case["stages"] * (cells * step_flops * steps + 2 * dense)}
    traces = -(-steps // case["every"]) if case["every"] else 0
    return {"bytes": cells * (step_bytes * steps + traces * (size[0] + size[1] * pots)),
            "flops": cells * (step_flops * steps + traces * per_stage)}


# ------------------------------------------------------------------ 64-bit values, plain torch
class _Lap(torch.autograd.Function):
    """The Laplacian on a cell list (symmetric, so it is its own transpose)."""

    @staticmethod
    def forward(ctx, psi, cells):
        ctx.cells = cells
        return cells.lap(psi)

    @staticmethod
    def backward(ctx, grad):
        return ctx.cells.lap(grad), None


class _Cells:
    """Active cells in ascending box order, their neighbours and packed slots."""

    def __init__(self, P, masks_of, stencil=7):
        nx, ny, nz = P.dims
        bx, by, bz = P.brick
        lin, vals = [], []
        for k0 in range(0, nz, 32):
            V, act = masks_of(k0, min(nz, k0 + 32))
            at = act.reshape(-1).nonzero().squeeze(1)
            lin.append(at + k0 * nx * ny)
            vals.append([v.reshape(-1)[at] for v in V])
        self.lin = torch.cat(lin)
        self.V = [torch.cat(v) for v in zip(*vals)]
        n = self.n = self.lin.numel()
        x, y, z = self.lin % nx, self.lin // nx % ny, self.lin // (nx * ny)
        nbx, nby = -(-nx // bx), -(-ny // by)
        brick = x // bx + nbx * (y // by + nby * (z // bz))
        seg = (x % bx + bx * (y % by + by * (z % bz))) // 4
        keys, inv = torch.unique(brick * (bx * by * bz // 4) + seg, return_inverse=True)
        self.slot = 4 * inv + x % 4
        self.n_packed = 4 * keys.numel()
        del keys, inv, brick, seg
        ih = [1.0 / s ** 2 for s in P.spacing]

        def neighbour(dx, dy, dz):
            ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz)
            want = self.lin + (dx + nx * (dy + ny * dz))
            at = torch.searchsorted(self.lin, want).clamp(max=n - 1)
            return torch.where(ok & (self.lin[at] == want), at, n)

        unit = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        coef = [ih[0], ih[1], ih[2]]
        centre = -2.0 * sum(ih)
        self.terms = []
        if stencil == 19:
            for a, b in ((0, 1), (0, 2), (1, 2)):
                w = (ih[a] + ih[b]) / 12.0
                coef[a] -= 2.0 * w
                coef[b] -= 2.0 * w
                centre += 4.0 * w
                for s in (1, -1):
                    for t in (1, -1):
                        d = [s * unit[a][i] + t * unit[b][i] for i in range(3)]
                        self.terms.append((w, neighbour(*d)))
        for a in range(3):
            for s in (1, -1):
                self.terms.append((coef[a], neighbour(*[s * v for v in unit[a]])))
        self.centre = centre

    def lap(self, psi):
        pad = torch.cat([psi, psi.new_zeros(1)])
        out = self.centre * psi
        for c, at in self.terms:
            out.add_(pad[at], alpha=c)
        return out

    def packed(self, v, fill=0.0):
        out = torch.full((self.n_packed,), fill, dtype=v.dtype, device=DEV)
        out[self.slot] = v
        return out


def _analytic_cells(P, case):
    x, y, z = (o + torch.arange(n, dtype=torch.float64, device=DEV) * s
               for n, s, o in zip(P.dims, P.spacing, P.origin))

    def masks(k0, k1):
        Z, Y, X = z[k0:k1, None, None], y[None, :, None], x[None, None, :]
        V, act = [], None
        for kind, p, cut in P.pots:
            if kind == "harmonic":
                v = 0.5 * (p[0] ** 2 * X * X + p[1] ** 2 * Y * Y + p[2] ** 2 * Z * Z)
            else:
                rho = torch.sqrt(X * X / p[1] ** 2 + Y * Y / p[2] ** 2 + Z * Z / p[3] ** 2)
                v = 0.5 * p[0] ** 2 * (rho - 1.0).square()
            V.append(v)
            act = v < cut if act is None else act | (v < cut)
        return V, act

    return _Cells(P, masks, case["stencil"])


def _start(P, C, case, seed, dtype):
    """The same initial state as prepare(), on the cell list, in 64 bits."""
    psi = _initial(P, C.packed(C.V[0], math.inf), case, seed, DTYPES[dtype][1])[C.slot]
    return psi.to(torch.complex128 if psi.is_complex() else torch.float64)


def _schedule(knots, t, T):
    n = len(knots)
    u = min(max(t / T * (n - 1), 0.0), n - 1.0)
    k = min(int(u), n - 2)
    return knots[k] + (u - k) * (knots[k + 1] - knots[k])


TABLEAUX = {
    "rk4": ([[], [1 / 2], [0, 1 / 2], [0, 0, 1]], [1 / 6, 1 / 3, 1 / 3, 1 / 6], [0, 1 / 2, 1 / 2, 1]),
    "rkhe3": ([[], [1 / 3], [0, 2 / 3]], [1 / 4, 0, 3 / 4], [0, 1 / 3, 2 / 3]),
    "rkck": ([[], [1 / 5], [3 / 40, 9 / 40], [3 / 10, -9 / 10, 6 / 5], [-11 / 54, 5 / 2, -70 / 27, 35 / 27],
              [1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096]],
             [37 / 378, 0, 250 / 621, 125 / 594, 0, 512 / 1771], [0, 1 / 5, 3 / 10, 3 / 5, 1, 7 / 8])}


def _rk_step(C, g, dt, psi, t, V_of, tableau):
    A, b, c = tableau
    ks = []
    for row, ci in zip(A, c):
        y = psi
        for a, k in zip(row, ks):
            if a:
                y = y + (dt * a) * k
        w = V_of(t + ci * dt) + g * (y.real.square() + y.imag.square())
        ks.append(-1j * (-0.5 * _Lap.apply(y, C) + w * y))
    out = psi
    for bi, k in zip(b, ks):
        if bi:
            out = out + (dt * bi) * k
    return out


def _imag_step(C, P, psi):
    dt, g = P.dt_imag, P.g
    E = torch.exp(-C.V[0] * dt / 2)
    psi = psi * E * (1 - g * psi.abs().square() * dt / 2)
    for _ in range(2):
        psi = psi + dt / 4 * C.lap(psi)
    psi = psi * E * (1 - g * psi.abs().square() * dt / 2)
    return psi * math.sqrt(N_ATOMS / (psi.abs().square().sum().item() * P.dV))


def _observables(C, P, psi, V):
    rho = psi.abs().square()
    norm = rho.sum().item() * P.dV
    kin = (-0.5 * (psi.conj() * C.lap(psi)).real).sum().item() * P.dV
    pot, inter = (V * rho).sum().item() * P.dV, (0.5 * P.g * rho.square()).sum().item() * P.dV
    o = {"norm": norm, "energy": kin + pot + inter, "mu": (kin + pot + 2 * inter) / norm, "e_kin": kin,
         "e_pot": pot, "e_int": inter}
    return [o[k] for k in OBS]


@torch.no_grad()
def exact(case, seed):
    P = _Problem(case)
    if case["kind"] == "stages":
        return _exact_stages(P, case, seed)
    if case["kind"] == "batch":
        psis, obs = [], []
        for i, Q in enumerate(_shells(case)):
            C = _analytic_cells(Q, case)
            psi = _start(Q, C, case, seed * 100 + i, case["dtype"])
            for _ in range(case["steps"]):
                psi = _imag_step(C, Q, psi)
            psis.append(C.packed(psi))
            obs.append(_observables(C, Q, psi, C.V[0]))
        return {"psi": psis, "obs": obs}
    C = _analytic_cells(P, case)
    psi = _start(P, C, case, seed, case["dtype"])
    if case["kind"] == "grad":
        return _exact_grad(P, C, case, seed, psi)
    if case["kind"] == "imag":
        for _ in range(case["steps"]):
            psi = _imag_step(C, P, psi)
        return {"psi": C.packed(psi), "obs": _observables(C, P, psi, C.V[0])}
    if case["geometry"] == "ramp":
        knots, T = _knots(seed), case["steps"] * P.dt_real

        def V_of(t):
            return torch.lerp(C.V[0], C.V[1], _schedule(knots, t, T))
    else:
        def V_of(t):
            return C.V[0]
    trace = []
    for n in range(case["steps"]):
        psi = _rk_step(C, P.g, P.dt_real, psi, n * P.dt_real, V_of, TABLEAUX[case["integrator"]])
        if case["every"] and ((n + 1) % case["every"] == 0 or n + 1 == case["steps"]):
            trace.append(_observables(C, P, psi, V_of((n + 1) * P.dt_real)))
    return {"psi": C.packed(psi), "trace": trace} if case["every"] else {"psi": C.packed(psi)}


def _exact_grad(P, C, case, seed, psi):
    from torch.utils.checkpoint import checkpoint
    target = _start(P, C, case, seed + 1, case["dtype"])
    T = case["steps"] * P.dt_real
    knots = torch.tensor(_knots(seed), dtype=torch.float32).to(DEV, torch.float64)
    with torch.enable_grad():
        knots.requires_grad_()

        def step(y, knots, t):
            return _rk_step(C, P.g, P.dt_real, y, t,
                            lambda u: C.V[0] + _schedule(knots, u, T) * (C.V[1] - C.V[0]), TABLEAUX["rk4"])

        for n in range(case["steps"]):
            psi = checkpoint(step, psi, knots, n * P.dt_real, use_reentrant=False)
        c = (target.conj() * psi).sum() * P.dV
        loss = 1.0 - (c.real.square() + c.imag.square())
        loss.backward()
    return {"loss": loss.item(), "grad": knots.grad, "psi": C.packed(psi.detach())}


def _exact_stages(P, case, seed):
    pots = _stage_potentials(case, P)
    mu = []
    for V in pots:  # sum over cells of max(mu - V, 0) dV / g = N, by sorting
        v = V.reshape(-1)
        v = torch.sort(v[v < 8.0 * P.mu0])[0].double()
        m = (P.g * N_ATOMS / P.dV + torch.cumsum(v, 0)) / torch.arange(1, v.numel() + 1, device=DEV)
        k = int((m > v).sum().item())  # the cells below mu are the first k
        mu.append(m[k - 1].item())
    dt = 0.5 * P.dt_real
    C0 = _Cells(P, lambda a, b: ([pots[0][a:b].double()], pots[0][a:b].double() < P.pots[0][2]))
    psi = _start(P, C0, case, seed, case["dtype"])
    lin, n_active, report = C0.lin, [], []
    del C0
    for i in range(case["stages"]):
        cut = 5.0 * max(mu[i], mu[i + 1])

        def masks(a, b):
            V = [pots[i][a:b].double(), pots[i + 1][a:b].double()]
            return V, (V[0] < cut) | (V[1] < cut)

        C = _Cells(P, masks)
        dense = psi.new_zeros(math.prod(P.dims))
        dense[lin] = psi
        psi, lin = dense[C.lin], C.lin
        del dense
        kept = psi.abs().square().sum().item() * P.dV
        T = case["steps"] * dt
        n = max(1, math.ceil(T / dt * (1.0 - 1e-12)))
        for j in range(n):
            psi = _rk_step(C, P.g, T / n, psi, j * T / n, lambda t: torch.lerp(C.V[0], C.V[1], t / T), TABLEAUX["rk4"])
        n_active.append(C.n)
        report.append([mu[i], mu[i + 1], cut, kept, psi.abs().square().sum().item() * P.dV])
    return {"psi": C.packed(psi), "n_active": n_active, "report": report}
