"""The tiles of the stencil kernels (runs of 128 stored segments with halo
lists) on masks that the shells do not give: isolated cells, half of all
cells, stripes whose every neighbour lies in another tile, fewer segments than
a tile, exactly one tile, one more; every brick shape, both stencils, every
state type.  Against the FP64 oracle: RK4 and imaginary-time steps and the
observables at the parity tolerances (1e-12 in FP64; a handful of FP32
roundings a step: 2e-6)."""
import math

import numpy as np
import pytest

import oracle
from gpu_cases import rel_l2
from paper_2603_05447_gb300 import gpe, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BRICKS = [(8, 8, 8), (8, 8, 4), (8, 4, 4)]
NPT = {gpe.GPE_C128: np.complex128, gpe.GPE_C64: np.complex64, gpe.GPE_R64: np.float64, gpe.GPE_R32: np.float32}


def mask_of(kind):
    rng = np.random.default_rng(11)
    if kind == "sparse":
        return rng.uniform(size=(37, 41, 83)) < 0.02
    if kind == "half":
        return rng.uniform(size=(21, 33, 45)) < 0.5
    if kind == "stripes":       # one segment of every second column, all rows and planes
        m = np.zeros((40, 48, 64), bool)
        m[:, :, 1::8] = True
        m[::3, 1::2, 6::16] = True
        return m
    if kind == "few":           # fewer segments than a tile
        m = np.zeros((9, 10, 21), bool)
        m[2:5, 3:7, 2:19] = True
        return m
    m = np.zeros((8, 8, 24), bool)
    m[:, :, :8] = True          # 128 segments: one tile of an 8x8x8 brick
    if kind == "one more":
        m[3, 4, 8] = True
    return m


MASKS = ["sparse", "half", "stripes", "few", "one tile", "one more"]


class Setup:
    def __init__(self, kind, dtype, brick, stencil):
        self.m = mask_of(kind)
        nz, ny, nx = self.m.shape
        self.h = (0.11, 0.1, 0.12)
        rng = np.random.default_rng(12)
        self.V = np.where(self.m, rng.uniform(0.0, 4.0, self.m.shape), 10.0)
        psi = np.where(self.m, rng.normal(size=self.m.shape) + 1j * rng.normal(size=self.m.shape), 0)
        if dtype in (gpe.GPE_R64, gpe.GPE_R32):
            psi = np.abs(psi) + 0j
        dV = math.prod(self.h)
        self.psi = inputs.normalise(psi, dV).astype(NPT[dtype] if dtype in (gpe.GPE_C128, gpe.GPE_C64) else complex)
        self.psi = self.psi.astype(np.complex128)
        self.og = oracle.Grid(self.m, self.h)
        self.g, self.dtype, self.stencil = 3.0, dtype, stencil
        lam = sum(2.0 / h ** 2 for h in self.h) + 10.0
        self.dt = 0.2 / lam
        self.grid = gpe.gpe_grid_create_dense(gpe.make_box(nx, ny, nz, *self.h), self.V, 5.0,
                                              gpe.make_opts(brick, stencil=stencil))
        self.st = gpe.gpe_state_create(self.grid, dtype)
        arr = self.psi.real if dtype in (gpe.GPE_R64, gpe.GPE_R32) else self.psi
        gpe.gpe_state_load(self.st, np.ascontiguousarray(arr.astype(NPT[dtype])), gpe.GPE_LAYOUT_DENSE)
        self.tol = 1e-12 if dtype in (gpe.GPE_C128, gpe.GPE_R64) else 2e-6

    def __enter__(self):
        return self

    def __exit__(self, *a):
        gpe.gpe_state_destroy(self.st)
        gpe.gpe_grid_destroy(self.grid)

    def dense(self):
        out = np.zeros(self.m.shape, NPT[self.dtype])
        gpe.gpe_state_store(self.st, out, gpe.GPE_LAYOUT_DENSE)
        return out.astype(np.complex128)


@pytest.mark.parametrize("stencil", [7, 19])
@pytest.mark.parametrize("brick", BRICKS)
@pytest.mark.parametrize("dtype", [gpe.GPE_C128, gpe.GPE_C64])
@pytest.mark.parametrize("kind", MASKS)
def test_rk4_on_odd_masks(kind, dtype, brick, stencil):
    with Setup(kind, dtype, brick, stencil) as S:
        V = S.og.compact(S.V)
        y = S.og.compact(S.dense())
        for _ in range(2):
            y = oracle.rk_step_np(S.og, V, y, S.g, 0.0, S.dt, stencil=stencil)
        gpe.gpe_step_real(S.st, gpe.real_params(S.g, S.dt), 2)
        assert rel_l2(S.og.compact(S.dense()), y) <= S.tol


@pytest.mark.parametrize("stencil", [7, 19])
@pytest.mark.parametrize("brick", BRICKS)
@pytest.mark.parametrize("dtype", [gpe.GPE_C128, gpe.GPE_C64, gpe.GPE_R64, gpe.GPE_R32])
@pytest.mark.parametrize("kind", MASKS)
def test_imaginary_time_and_observables_on_odd_masks(kind, dtype, brick, stencil):
    with Setup(kind, dtype, brick, stencil) as S:
        V = S.og.compact(S.V)
        y = S.og.compact(S.dense())
        for _ in range(2):
            y, _ = oracle.itp_step_np(S.og, V, y, S.g, S.dt, stencil=stencil)
        gpe.gpe_step_imag(S.st, gpe.gpe_imag_params(S.g, S.dt, 1.0), 2)
        got = S.og.compact(S.dense())
        assert rel_l2(got, y) <= S.tol
        o, ref = gpe.gpe_observables(S.st, S.g), oracle.observables_np(S.og, V, S.g, got, stencil=stencil)
        for k in ("norm", "energy", "mu", "e_kin", "e_pot", "e_int"):
            assert abs(o[k] - ref[k]) <= S.tol * max(abs(ref[k]), abs(ref["energy"])), k


@pytest.mark.parametrize("integrator", ["RKHE3", "RKCK"])
@pytest.mark.parametrize("dtype", [gpe.GPE_C128, gpe.GPE_C64])
@pytest.mark.parametrize("kind", ["sparse", "half", "one more"])
def test_general_integrators_on_odd_masks(kind, dtype, integrator):
    with Setup(kind, dtype, (8, 8, 4), 7) as S:
        V = S.og.compact(S.V)
        y = S.og.compact(S.dense())
        for _ in range(2):
            y = oracle.rk_step_np(S.og, V, y, S.g, 0.0, S.dt, method=integrator)
        gpe.gpe_step_real(S.st, gpe.real_params(S.g, S.dt, integrator=getattr(gpe, "GPE_" + integrator)), 2)
        assert rel_l2(S.og.compact(S.dense()), y) <= S.tol


# Sums of a block are put into FP64 every 64 tiles.  All-active boxes of bricks
# of 128 segments (one tile each) around 64 tiles a block on 152 SMs with five
# to eight blocks an SM, where only some blocks reach the 64th.
@pytest.mark.parametrize("nb", [(40, 40, 30), (40, 40, 36), (40, 50, 29), (40, 40, 42), (40, 50, 34), (45, 48, 36)])
@pytest.mark.parametrize("dtype", [gpe.GPE_C64, gpe.GPE_R32])
def test_sums_over_sixty_odd_tiles_a_block(nb, dtype):
    h = 0.1
    box = gpe.make_box(8 * nb[0], 8 * nb[1], 8 * nb[2], h)
    grid = gpe.gpe_grid_create_analytic(box, gpe.make_potential(gpe.GPE_POT_HARMONIC, 1e-3, 1e-3, 1e-3), 1e9)
    st = gpe.gpe_state_create(grid, dtype)
    try:
        n = 512 * nb[0] * nb[1] * nb[2]
        gen = torch.Generator(device="cuda").manual_seed(5)
        re = torch.rand(n, generator=gen, device="cuda") + 0.5
        psi = re if dtype == gpe.GPE_R32 else torch.complex(re, 0.3 * re)
        gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_COMPACT)
        want = float(psi.abs().double().square().sum()) * h ** 3
        assert abs(gpe.gpe_observables(st, 0.1)["norm"] - want) <= 1e-6 * want
        gpe.gpe_step_imag(st, gpe.gpe_imag_params(0.1, 1e-4, 2.0), 2)
        assert abs(gpe.gpe_observables(st, 0.1)["norm"] - 2.0) <= 2e-6
    finally:
        gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(grid)


def neighbours(psi):
    """Opposite-neighbour sums along x, y, z; zero outside."""
    p = np.pad(psi, 1)
    return (p[1:-1, 1:-1, :-2] + p[1:-1, 1:-1, 2:], p[1:-1, :-2, 1:-1] + p[1:-1, 2:, 1:-1],
            p[:-2, 1:-1, 1:-1] + p[2:, 1:-1, 1:-1])


@pytest.mark.parametrize("spacing", [(0.1, 0.1, 0.1), (0.1, 0.105, 0.097), (0.1, 0.1, 30.0), (1e-9, 2e-9, 3e-9)])
@pytest.mark.parametrize("decades", [0, 12, 40, 300])
def test_double_sums_in_fixed_point(spacing, decades):
    """One imaginary-time step (two Euler substeps, V = 0 and g = 0) of complex128 values over
    many orders of magnitude, zeros and denormals among them, against the same
    in extended precision: the error of every cell stays within the rounding
    of FP64 on the sum of the magnitudes that enter it (12 roundings a
    substep, 4 for the factors)."""
    rng = np.random.default_rng(7)
    shape = (9, 10, 21)
    psi = (rng.normal(size=shape) + 1j * rng.normal(size=shape)) * 10.0 ** -rng.uniform(0, decades, shape)
    psi[rng.uniform(size=shape) < 0.1] = 0.0
    psi[2:7, 3:8, 4:15] = 0.0
    psi[4, 5, 6], psi[4, 5, 7] = 3e-310, 1e-290j
    h = [np.longdouble(s) for s in spacing]
    dt = 0.4 * float(min(h)) ** 2
    box = gpe.make_box(shape[2], shape[1], shape[0], *spacing)
    grid = gpe.gpe_grid_create_dense(box, np.zeros(shape), 1.0)
    st = gpe.gpe_state_create(grid, gpe.GPE_C128)
    out = np.empty_like(psi)
    try:
        gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_DENSE)
        gpe.gpe_step_imag(st, gpe.gpe_imag_params(0.0, dt, 1.0), 1)
        gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
    finally:
        gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(grid)
    for part, got in ((psi.real, out.real), (psi.imag, out.imag)):
        want, size = part.astype(np.longdouble), np.abs(part).astype(np.longdouble)
        for _ in range(2):
            lap, mag = -2 * sum(1 / s ** 2 for s in h) * want, 2 * sum(1 / s ** 2 for s in h) * size
            for n, m, s in zip(neighbours(want), neighbours(size), h):
                lap, mag = lap + n / s ** 2, mag + m / s ** 2
            want, size = want + dt / 4 * lap, size + dt / 4 * mag
        scale = np.vdot(got.astype(np.longdouble), want) / np.vdot(want, want)  # the renormalisation
        assert np.all(np.abs(got - scale * want) <= 28 * 2.0 ** -53 * scale * size + 1e-307 * scale)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_a_value_that_is_not_finite_reaches_its_neighbours(bad):
    shape = (5, 6, 9)
    box = gpe.make_box(9, 6, 5, 0.1)
    grid = gpe.gpe_grid_create_dense(box, np.zeros(shape), 1.0)
    st = gpe.gpe_state_create(grid, gpe.GPE_C128)
    psi = np.ones(shape, np.complex128)
    psi[2, 3, 4] = bad
    out = np.empty_like(psi)
    try:
        gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_DENSE)
        gpe.gpe_step_real(st, gpe.real_params(0.0, 1e-4), 1)
        gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
    finally:
        gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(grid)
    for k, j, i in ((2, 3, 4), (1, 3, 4), (2, 2, 4), (2, 3, 3), (2, 3, 5)):
        assert not np.isfinite(out[k, j, i])
