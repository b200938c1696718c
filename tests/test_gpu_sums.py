"""The FP64 sums of single-precision terms (norm, observables, batch sums, knot
derivative) where the terms are so large that a float cannot hold a few hundred
of them, though FP64 holds their sum.  With g = 0 every quantity is a power of
the state's scale, and scaling by a power of two is exact in the terms: the
scaled run's results are the unscaled run's times that power, up to the sums'
own rounding (a pair of floats is good to 2^-48 a term, at most 2048 terms
before FP64: 1e-11).  The renormalisation factor is rounded to a float, so after
a step the two states may differ by a handful of FP32 roundings (2e-6)."""
import numpy as np
import pytest

from gpu_cases import rel_l2
from paper_2603_05447_gb300 import gpe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, H = 48, 2.0
K = 61                       # |psi|^2 grows by 2^122: up to 1.2e37 a cell, 5e37 a segment
TERMS, STEPS = 1e-11, 2e-6
ATOMS = 1e6                  # the size of the state before the first step
REAL = (gpe.GPE_R64, gpe.GPE_R32)
NP = {gpe.GPE_C64: np.complex64, gpe.GPE_R32: np.float32}


def start(dtype, n=N):
    rng = np.random.default_rng(3)
    psi = rng.uniform(0.5, 1.0, (n, n, n))
    if dtype not in REAL:
        psi = psi + 1j * rng.uniform(0.5, 1.0, psi.shape)
    return psi.astype(NP[dtype]), rng.uniform(0.0, 2.0, psi.shape)


class Box:
    def __init__(self, dtype, V, stencil=7, V1=None):
        n = V.shape[0]
        box = gpe.make_box(n, n, n, H)
        self.grid = gpe.gpe_grid_create_dense(box, V, 1e9, gpe.make_opts((8, 8, 8), stencil=stencil))
        if V1 is not None:
            gpe.gpe_grid_set_potential(self.grid, 1, V1)
        self.states, self.dtype, self.shape = [], dtype, V.shape

    def state(self, psi):
        self.states.append(gpe.gpe_state_create(self.grid, self.dtype))
        gpe.gpe_state_load(self.states[-1], psi, gpe.GPE_LAYOUT_DENSE)
        return self.states[-1]

    def dense(self, st):
        out = np.zeros(self.shape, NP[self.dtype])
        gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
        return out.astype(np.complex128)

    def __enter__(self):
        return self

    def __exit__(self, *a):
        for st in self.states:
            gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(self.grid)


def same_up_to_scale(big, small):
    for k in ("norm", "e_kin", "e_pot", "energy"):
        assert abs(big[k] / 4.0 ** K - small[k]) <= TERMS * (abs(small[k]) + small["norm"]), k
    assert big["e_int"] == 0.0 and big["nonfinite"] == 0


@pytest.mark.parametrize("stencil", [7, 19])
@pytest.mark.parametrize("dtype", [gpe.GPE_C64, gpe.GPE_R32])
def test_observables_and_norm_of_large_values(dtype, stencil):
    psi, V = start(dtype)
    with Box(dtype, V, stencil) as B:
        a, b = B.state(psi), B.state(psi * np.float32(2.0 ** K))
        same_up_to_scale(gpe.gpe_observables(b, 0.0), gpe.gpe_observables(a, 0.0))
        for st, N_ in ((a, ATOMS), (b, ATOMS * 4.0 ** K)):
            gpe.gpe_step_imag(st, gpe.gpe_imag_params(0.0, 0.1, N_), 2)
        assert rel_l2(B.dense(b) / 2.0 ** K, B.dense(a)) <= STEPS


@pytest.mark.parametrize("dtype", [gpe.GPE_C64, gpe.GPE_R32])
def test_batch_sums_of_large_values(dtype):
    psi, V = start(dtype)
    with Box(dtype, V) as B:
        st = [B.state(psi), B.state(psi * np.float32(2.0 ** K))]
        batch = gpe.gpe_batch_create(st)
        try:
            p = [gpe.gpe_imag_params(0.0, 0.1, ATOMS * 4.0 ** k) for k in (0, K)]
            _, _, _, obs = gpe.gpe_batch_ground_state(batch, p, 1e-12, 2, 2, check=False)
        finally:
            gpe.gpe_batch_destroy(batch)
        for k in ("norm", "e_kin", "e_pot"):
            assert abs(obs[1][k] / 4.0 ** K - obs[0][k]) <= 2 * STEPS * (abs(obs[0][k]) + obs[0]["norm"]), k
        assert rel_l2(B.dense(st[1]) / 2.0 ** K, B.dense(st[0])) <= STEPS


def test_knot_derivative_of_large_terms():
    """A target of 2^53 times the size: the adjoint starts from -2 dV <t|psi> t, about
    2e38, and a cell's term of the knot derivative reaches about 5e36."""
    n, dt, steps = 32, 0.02, 20
    rng = np.random.default_rng(4)
    V1 = np.broadcast_to(6.0 * np.arange(n)[:, None, None] / (n - 1), (n, n, n)).copy()
    psi = np.exp(0.1j * rng.normal(size=V1.shape)).astype(np.complex64)
    got = []
    with Box(gpe.GPE_C64, np.zeros_like(V1), V1=V1) as B:
        p = gpe.real_params(0.0, dt, gpe.GPE_V_BLEND, [0.9, 1.0, 0.8], steps * dt)
        for k in (0, 53):
            st, target = B.state(psi), B.state(psi * np.float32(0.8 * 2.0 ** k))
            tape = gpe.gpe_ramp_forward(st, p, steps, 0.0, 7)
            try:
                loss, grad = gpe.gpe_ramp_backward(tape, target, 3)
            finally:
                gpe.gpe_tape_destroy(tape)
            got.append(((1.0 - loss) / 4.0 ** k, np.array(grad) / 4.0 ** k))
    (c0, g0), (c1, g1) = got
    assert abs(c1 - c0) <= 1e-12 * (1.0 + c0)  # 1 - loss of the unscaled run rounds at 1
    assert np.all(np.isfinite(g1)) and np.abs(g1 - g0).max() <= TERMS * np.abs(g0).max()
