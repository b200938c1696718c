"""The steps commute exactly with psi -> -psi and keep a state that is exactly
odd under a mirror exactly odd, as FP64 arithmetic does: every operation rounds
opposite values to opposite results.  Unequal spacings, whose neighbour sums in
double precision go through fractions of the largest coefficient; every
schedule, both stencils.  (The 19-point stencil adds its four y-z edges one after
the other, so only its mirror along x swaps equal sums.)"""
import numpy as np
import pytest

from paper_2603_05447_gb300 import gpe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPACING = (0.1, 0.105, 0.097)
SHAPE = (19, 22, 24)          # z, y, x
SCHEDS = [(gpe.GPE_SCHED_STAGED, 7), (gpe.GPE_SCHED_STAGED, 19), (gpe.GPE_SCHED_WAVE, 7), (gpe.GPE_SCHED_WAVE2, 7),
          (gpe.GPE_SCHED_PAIR, 7)]


def stepped(psi, V, kind, sched, stencil, g):
    dtype = {np.dtype(np.complex128): gpe.GPE_C128, np.dtype(np.float64): gpe.GPE_R64}[psi.dtype]
    box = gpe.make_box(SHAPE[2], SHAPE[1], SHAPE[0], *SPACING)
    grid = gpe.gpe_grid_create_dense(box, V, 1e9, gpe.make_opts((8, 8, 4), sched=sched, stencil=stencil))
    st = gpe.gpe_state_create(grid, dtype)
    out = np.empty_like(psi)
    try:
        gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_DENSE)
        if kind == "real":
            gpe.gpe_step_real(st, gpe.real_params(g, 2e-4), 3)
        else:
            gpe.gpe_step_imag(st, gpe.gpe_imag_params(g, 2e-3, 1.0), 3)
        gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
    finally:
        gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(grid)
    return out


CASES = [("real", np.complex128), ("imag", np.complex128), ("imag", np.float64)]


@pytest.mark.parametrize("sched,stencil", SCHEDS)
@pytest.mark.parametrize("kind,dtype", CASES)
def test_opposite_states_stay_opposite(kind, dtype, sched, stencil):
    rng = np.random.default_rng(6)
    psi = rng.normal(size=SHAPE)
    if dtype == np.complex128:
        psi = psi + 1j * rng.normal(size=SHAPE)
    V = rng.uniform(0.0, 3.0, SHAPE)
    a, b = (stepped(p, V, kind, sched, stencil, 2.0) for p in (psi, -psi))
    assert np.array_equal(a, -b)


@pytest.mark.parametrize("sched,stencil,axis", [(s, n, a) for s, n in SCHEDS for a in (0, 1, 2) if n == 7 or a == 2])
@pytest.mark.parametrize("kind,dtype", CASES)
def test_an_odd_state_stays_odd(kind, dtype, sched, stencil, axis):
    rng = np.random.default_rng(8)
    psi = rng.normal(size=SHAPE)
    if dtype == np.complex128:
        psi = psi + 1j * rng.normal(size=SHAPE)
    psi = psi - np.flip(psi, axis)
    V = rng.uniform(0.0, 3.0, SHAPE)
    V = V + np.flip(V, axis)
    out = stepped(psi, V, kind, sched, stencil, 2.0)
    assert np.array_equal(out, -np.flip(out, axis))
