"""Double precision on boxes whose spacings differ by more than the fixed-point
neighbour sums serve (a factor sqrt 8), just below and far above: the kernels'
FP64 instances against the FP64 oracle at the parity tolerance (1e-12), and the
schedules' identical bits in real time."""
import numpy as np
import pytest

import oracle
from gpu_cases import rel_l2
from paper_2603_05447_gb300 import gpe, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (13, 18, 23)
SPACINGS = [(0.1, 0.1, 0.28), (0.1, 0.1, 0.1 * 8 ** 0.5), (0.1, 0.1, 0.2829), (0.1, 0.31, 0.1), (0.9, 0.1, 0.11)]
TOL = 1e-12
G = 2.0


class Case:
    def __init__(self, h):
        rng = np.random.default_rng(5)
        self.h, self.V = h, rng.uniform(0.0, 3.0, SHAPE)
        self.mask = rng.uniform(size=SHAPE) < 0.8
        self.V[~self.mask] = 10.0
        psi = np.where(self.mask, rng.normal(size=SHAPE) + 1j * rng.normal(size=SHAPE), 0)
        self.psi = inputs.normalise(psi, float(np.prod(h)))
        self.og = oracle.Grid(self.mask, h)
        self.dt = 0.2 / (sum(2.0 / s ** 2 for s in h) + 6.0)

    def run(self, dtype, step, sched=gpe.GPE_SCHED_STAGED):
        box = gpe.make_box(SHAPE[2], SHAPE[1], SHAPE[0], *self.h)
        grid = gpe.gpe_grid_create_dense(box, self.V, 5.0, gpe.make_opts((8, 8, 4), sched=sched))
        st = gpe.gpe_state_create(grid, dtype)
        psi = self.psi if dtype == gpe.GPE_C128 else np.ascontiguousarray(np.abs(self.psi))
        out = np.zeros_like(psi)
        try:
            gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_DENSE)
            step(st)
            gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
        finally:
            gpe.gpe_state_destroy(st)
            gpe.gpe_grid_destroy(grid)
        return out


@pytest.mark.parametrize("h", SPACINGS)
@pytest.mark.parametrize("integrator", ["RK4", "RKHE3", "RKCK"])
def test_real_time(h, integrator):
    c = Case(h)
    V, y = c.og.compact(c.V), c.og.compact(c.psi)
    for _ in range(3):
        y = oracle.rk_step_np(c.og, V, y, G, 0.0, c.dt, method=integrator)
    p = gpe.real_params(G, c.dt, integrator=getattr(gpe, "GPE_" + integrator))
    out = c.run(gpe.GPE_C128, lambda st: gpe.gpe_step_real(st, p, 3))
    assert rel_l2(c.og.compact(out), y) <= TOL
    if integrator == "RK4":
        for sched in (gpe.GPE_SCHED_WAVE, gpe.GPE_SCHED_WAVE2, gpe.GPE_SCHED_PAIR):
            assert np.array_equal(c.run(gpe.GPE_C128, lambda st: gpe.gpe_step_real(st, p, 3), sched), out)


@pytest.mark.parametrize("h", SPACINGS)
@pytest.mark.parametrize("dtype,sched", [(gpe.GPE_C128, gpe.GPE_SCHED_STAGED), (gpe.GPE_R64, gpe.GPE_SCHED_STAGED),
                                         (gpe.GPE_C128, gpe.GPE_SCHED_WAVE), (gpe.GPE_C128, gpe.GPE_SCHED_PAIR)])
def test_imaginary_time(h, dtype, sched):
    c = Case(h)
    V, y = c.og.compact(c.V), c.og.compact(c.psi if dtype == gpe.GPE_C128 else np.abs(c.psi) + 0j)
    for _ in range(3):
        y, _ = oracle.itp_step_np(c.og, V, y, G, c.dt)
    out = c.run(dtype, lambda st: gpe.gpe_step_imag(st, gpe.gpe_imag_params(G, c.dt, 1.0), 3), sched)
    assert rel_l2(c.og.compact(out + 0j), y) <= TOL
