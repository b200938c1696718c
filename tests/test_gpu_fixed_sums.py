"""The neighbour sums of the double-precision passes in 64-bit fixed point, seen
by themselves: a state whose real part is zero gets, in one RK4 step so short that
its stages do not differ, a real part of dt times minus half the Laplacian of
its imaginary part.  Cells whose opposite neighbours cancel exactly and leave
sums of many sizes show the sums' absolute error: six cuts and three products
of at most 2^-59 of the largest neighbour (times the largest 1/h^2); beside it
FP64 rounds at 2^-53 of the sum and of the centre's term, ten times at most.  In
exact rational arithmetic."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2603_05447_gb300 import gpe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (14, 17, 21)
DT = 2.0 ** -70


def planted(decades):
    """Random cells; every fourth one is 0 or small, with an opposite pair of size 1
    along a random axis and the other four neighbours up to `decades` smaller."""
    rng = np.random.default_rng(17)
    psi = rng.normal(size=SHAPE)
    cells = [(k, j, i) for k in range(1, SHAPE[0] - 1, 3) for j in range(1, SHAPE[1] - 1, 3) for i in range(1, SHAPE[2] - 1, 3)]
    for n, (k, j, i) in enumerate(cells):
        axis, size = n % 3, 10.0 ** -rng.uniform(0, decades)
        psi[k, j, i] = 0.0 if n % 2 else size * rng.normal()
        for a, (dk, dj, di) in enumerate(((1, 0, 0), (0, 1, 0), (0, 0, 1))):
            v = rng.normal()
            for s in (1, -1):
                psi[k + s * dk, j + s * dj, i + s * di] = s * v if a == axis else size * rng.normal()
    return psi, cells


@pytest.mark.parametrize("sched", [gpe.GPE_SCHED_STAGED, gpe.GPE_SCHED_WAVE, gpe.GPE_SCHED_PAIR])
@pytest.mark.parametrize("spacing", [(0.125, 0.125, 0.125), (0.1, 0.105, 0.097), (0.1, 0.2, 0.25)])
@pytest.mark.parametrize("decades", [0, 8, 16, 30])
def test_sums_whose_largest_terms_cancel(spacing, decades, sched):
    psi, cells = planted(decades)
    box = gpe.make_box(SHAPE[2], SHAPE[1], SHAPE[0], *spacing)
    grid = gpe.gpe_grid_create_dense(box, np.zeros(SHAPE), 1.0, gpe.make_opts((8, 8, 4), sched=sched))
    st = gpe.gpe_state_create(grid, gpe.GPE_C128)
    out = np.empty(SHAPE, np.complex128)
    try:
        gpe.gpe_state_load(st, 1j * psi, gpe.GPE_LAYOUT_DENSE)
        gpe.gpe_step_real(st, gpe.real_params(0.0, DT), 1)
        gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
    finally:
        gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(grid)
    c = [Fraction(1.0 / (h * h)) for h in spacing]  # the doubles that the step computes with
    ulp, cut = Fraction(2) ** -53, Fraction(2) ** -59
    for k, j, i in cells:
        n = [Fraction(psi[k, j, i - 1]), Fraction(psi[k, j, i + 1]), Fraction(psi[k, j - 1, i]), Fraction(psi[k, j + 1, i]),
             Fraction(psi[k - 1, j, i]), Fraction(psi[k + 1, j, i])]
        s = c[0] * (n[0] + n[1]) + c[1] * (n[2] + n[3]) + c[2] * (n[4] + n[5])
        centre = 2 * sum(c) * Fraction(psi[k, j, i])
        bound = 9 * cut * max(c) * max(abs(v) for v in n) + 10 * ulp * (abs(s) + abs(centre))
        got = Fraction(float(out.real[k, j, i])) / Fraction(DT)
        assert abs(got + (s - centre) / 2) <= bound / 2
