"""A potential replaced between calls: imaginary-time steps and ground states of
a state that has stepped on the old one equal those of a fresh state bit for
bit (the propagator table is made again), every state type, stencil and
schedule; replacing slot 1 changes nothing."""
import numpy as np
import pytest

from paper_2603_05447_gb300 import gpe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (17, 20, 23)
NPT = {gpe.GPE_C128: np.complex128, gpe.GPE_C64: np.complex64, gpe.GPE_R64: np.float64, gpe.GPE_R32: np.float32}
P = gpe.gpe_imag_params(3.0, 1e-3, 1.0)


def stepped(st, psi, steps=5):
    gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_DENSE)
    gpe.gpe_step_imag(st, P, steps)
    out = np.zeros_like(psi)
    gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
    return out


@pytest.mark.parametrize("dtype", list(NPT))
@pytest.mark.parametrize("sched,stencil", [(gpe.GPE_SCHED_STAGED, 7), (gpe.GPE_SCHED_STAGED, 19),
                                           (gpe.GPE_SCHED_WAVE, 7), (gpe.GPE_SCHED_PAIR, 7)])
def test_imaginary_time_after_a_new_potential(dtype, sched, stencil):
    rng = np.random.default_rng(2)
    V, W = rng.uniform(0.0, 5.0, SHAPE), rng.uniform(0.0, 500.0, SHAPE)
    psi = rng.uniform(0.5, 1.0, SHAPE).astype(NPT[dtype])
    box = gpe.make_box(SHAPE[2], SHAPE[1], SHAPE[0], 0.1)
    grid = gpe.gpe_grid_create_dense(box, V, 1e9, gpe.make_opts((8, 8, 4), sched=sched, stencil=stencil))
    used, fresh = gpe.gpe_state_create(grid, dtype), gpe.gpe_state_create(grid, dtype)
    try:
        old = stepped(used, psi)
        gpe.gpe_grid_set_potential(grid, 1, W)
        assert np.array_equal(stepped(used, psi), old)
        gpe.gpe_grid_set_potential(grid, 0, W)
        new = stepped(used, psi)
        assert not np.array_equal(new, old)
        assert np.array_equal(new, stepped(fresh, psi))
        mu = []
        for st in (used, fresh):
            gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_DENSE)
            mu.append(gpe.gpe_ground_state(st, P, 1e9, 20, 40))
        assert mu[0] == mu[1]
    finally:
        gpe.gpe_state_destroy(used)
        gpe.gpe_state_destroy(fresh)
        gpe.gpe_grid_destroy(grid)
