"""The ramp gradient where cells of the region have V0 = +inf (a wall inside it):
psi is zero there after a step, so neither the loss nor the gradient may depend
on what the target holds there.  Both runs do the same arithmetic: equal bits."""
import numpy as np
import pytest

from paper_2603_05447_gb300 import gpe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, STEPS = 20, 6


@pytest.mark.parametrize("K", [2, STEPS])
@pytest.mark.parametrize("dtype", [gpe.GPE_C64, gpe.GPE_C128])
def test_target_values_at_walls_do_not_matter(dtype, K):
    rng = np.random.default_rng(6)
    cdt = np.complex128 if dtype == gpe.GPE_C128 else np.complex64
    shape = (N, N, N)
    V0, V1 = rng.uniform(0.0, 2.0, shape), rng.uniform(0.0, 4.0, shape)
    wall = rng.uniform(size=shape) < 0.2
    V0[wall] = np.inf
    psi, target = (rng.normal(size=shape) + 1j * rng.normal(size=shape) for _ in range(2))
    target += 2.0 * psi  # so that they overlap
    grid = gpe.gpe_grid_create_dense(gpe.make_box(N, N, N, 0.5), np.zeros(shape), 1.0)
    gpe.gpe_grid_set_potential(grid, 0, V0)
    gpe.gpe_grid_set_potential(grid, 1, V1)
    p = gpe.real_params(0.5, 0.01, gpe.GPE_V_BLEND, [0.2, 0.9, 0.4], STEPS * 0.01)
    st = gpe.gpe_state_create(grid, dtype)
    tg = gpe.gpe_state_create(grid, dtype)
    tape, got = None, []
    try:
        gpe.gpe_state_load(st, (psi / N ** 1.5).astype(cdt), gpe.GPE_LAYOUT_DENSE)
        tape = gpe.gpe_ramp_forward(st, p, STEPS, 0.0, K)
        for t in (target, np.where(wall, 0, target)):
            gpe.gpe_state_load(tg, (t / N ** 1.5).astype(cdt), gpe.GPE_LAYOUT_DENSE)
            loss, grad = gpe.gpe_ramp_backward(tape, tg, 3)
            got.append((loss, *np.asarray(grad)))
    finally:
        if tape is not None:
            gpe.gpe_tape_destroy(tape)
        gpe.gpe_state_destroy(st)
        gpe.gpe_state_destroy(tg)
        gpe.gpe_grid_destroy(grid)
    assert got[0] == got[1] and np.all(np.isfinite(got[1])) and got[1][1] != 0.0
