"""The ramp gradient on both sides of the tape's memory rule (the stage states of
a segment are kept where they take at most an eighth of the free memory): one
segment so long that they do not, against short ones that do.  dt is a power of
two, so every stage time is exact and both runs do the same arithmetic: equal
bits."""
import numpy as np
import pytest

from paper_2603_05447_gb300 import gpe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, DT = 64, 2.0 ** -7


def test_gradient_without_kept_stage_states():
    rng = np.random.default_rng(2)
    shape = (N, N, N)
    V0, V1 = rng.uniform(0.0, 1.0, shape), rng.uniform(0.0, 2.0, shape)
    psi, target = ((rng.normal(size=shape) + 1j * rng.normal(size=shape)) / N ** 1.5 for _ in range(2))
    target = target + psi
    grid = gpe.gpe_grid_create_dense(gpe.make_box(N, N, N, 1.0), V0, 1e9)
    gpe.gpe_grid_set_potential(grid, 1, V1)
    copy = N ** 3 * 8  # bytes of a state
    steps = torch.cuda.mem_get_info()[0] // (24 * copy) + 100  # 3 steps copies > free / 8
    p = gpe.real_params(0.5, DT, gpe.GPE_V_BLEND, [0.2, 0.9, 0.4, 0.8], steps * DT)
    st = gpe.gpe_state_create(grid, gpe.GPE_C64)
    tg = gpe.gpe_state_create(grid, gpe.GPE_C64)
    got, free = [], []
    try:
        gpe.gpe_state_load(tg, target.astype(np.complex64), gpe.GPE_LAYOUT_DENSE)
        for K in (steps, 100):
            gpe.gpe_state_load(st, psi.astype(np.complex64), gpe.GPE_LAYOUT_DENSE)
            before = torch.cuda.mem_get_info()[0]
            tape = gpe.gpe_ramp_forward(st, p, steps, 0.0, K)
            try:
                free.append(before - torch.cuda.mem_get_info()[0])
                loss, grad = gpe.gpe_ramp_backward(tape, tg, 4)
            finally:
                gpe.gpe_tape_destroy(tape)
            got.append((loss, *np.asarray(grad)))
    finally:
        gpe.gpe_state_destroy(st)
        gpe.gpe_state_destroy(tg)
        gpe.gpe_grid_destroy(grid)
    assert free[0] < 2 * steps * copy  # one copy a step, not four
    assert free[1] > (-(-steps // 100) + 350) * copy  # checkpoints and four copies of a segment
    assert got[0] == got[1] and np.all(np.isfinite(got[0])) and got[0][2] != 0.0
