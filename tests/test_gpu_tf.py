"""Thomas-Fermi mu on the GPU against the root found by sorting, at the sizes
and inputs where the passes over a dense box can go wrong: fewer cells than a
vector load, remainders, unaligned device arrays, FP32 and FP64, sets that
hold one cell or every cell, walls at +inf, negative potentials and boxes
above and below the sample's size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2603_05447_gb300 import gpe  # noqa: E402


def root(V, target):
    """The mu with sum max(mu - V, 0) = target, from the sorted finite cells."""
    v = np.sort(V[V < np.inf].astype(np.float64).ravel())
    m = (target + np.cumsum(v)) / np.arange(1, v.size + 1)
    k = int((m > v).sum())
    return m[k - 1]


def potential(shape, kind):
    rng = np.random.default_rng(sum(shape))
    z, y, x = np.meshgrid(*[np.linspace(-1, 1, n) if n > 1 else np.zeros(1) for n in shape], indexing="ij")
    if kind == "shell":
        return 500.0 * (np.sqrt(x * x + 1.1 * y * y + 1.3 * z * z) - 0.7) ** 2
    if kind == "negative":
        return -50.0 + 30.0 * (x * x + y * y + z * z)
    if kind == "flat":
        return np.full(shape, 2.5)
    V = rng.uniform(0.0, 10.0, shape)          # "walls"
    V[rng.uniform(size=shape) < 0.3] = np.inf
    V.ravel()[0] = 0.5
    return V


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 3), (5, 7, 9), (31, 33, 37), (64, 64, 64), (97, 101, 103)])
@pytest.mark.parametrize("kind", ["shell", "negative", "flat", "walls"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("offset", [0, 1])
def test_tf_mu_is_the_root(shape, kind, dtype, offset):
    h = 0.1
    box = gpe.make_box(shape[2], shape[1], shape[0], h)
    V = potential(shape, kind).astype(dtype)
    buf = torch.empty(V.size + offset, dtype=torch.from_numpy(V).dtype, device="cuda")
    dV = buf[offset:]
    dV.copy_(torch.from_numpy(V.ravel()))
    for gN in (1e-6 * h ** 3, 1.0 * h ** 3, 50.0 * V.size * h ** 3):  # a cell or few, some, every cell
        want = root(V, gN / h ** 3)
        got = gpe.gpe_tf_mu_dense(box, dV, gN, 1.0)
        # FP64 sums of at most 1e6 terms of one size: n eps / 2 in the worst case, far less in practice
        assert abs(got - want) <= 1e-11 * max(abs(want), 60.0)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_tf_mu_refuses_a_potential_without_a_finite_root(bad):
    V = np.full((8, 8, 8), bad)
    with pytest.raises(gpe.GpeError):
        gpe.gpe_tf_mu_dense(gpe.make_box(8, 8, 8, 0.1), V, 1.0, 1.0)
    if bad == -np.inf:
        V = np.ones((8, 8, 8))
        V[3, 4, 5] = bad
        with pytest.raises(gpe.GpeError):
            gpe.gpe_tf_mu_dense(gpe.make_box(8, 8, 8, 0.1), V, 1.0, 1.0)


@pytest.mark.parametrize("dtype", [np.float64])
def test_tf_mu_sum_that_overflows_is_refused(dtype):
    V = np.ones((8, 8, 8), dtype)
    V[:4] = 1e307
    with pytest.raises(gpe.GpeError):
        gpe.gpe_tf_mu_dense(gpe.make_box(8, 8, 8, 0.1), V, 1.0, 1.0)


def test_tf_mu_of_large_fp32_cells_is_the_root():
    V = potential((33, 34, 35), "shell").astype(np.float32)
    V[::3] = 2e37  # a thread's float pair would not hold their sum
    h, target = 0.1, 1e42
    got = gpe.gpe_tf_mu_dense(gpe.make_box(35, 34, 33, h), V, target * h ** 3, 1.0)
    want = root(V, target)
    assert abs(got - want) <= 1e-11 * want


@pytest.mark.parametrize("kind", ["harmonic", "shell"])
def test_tf_mu_analytic_outside_the_range_of_fp32(kind):
    n, h = 24, 1e-26
    x = (np.arange(n) - (n - 1) / 2) * h
    r2 = x[:, None, None] ** 2 + x[:, None] ** 2 + x ** 2
    if kind == "harmonic":
        w = 1e26
        V, pot = 0.5 * w * w * r2, gpe.make_potential(gpe.GPE_POT_HARMONIC, w, w, w)
    else:
        w, a = 30.0, 7 * h
        V, pot = 0.5 * w * w * (np.sqrt(r2 / a ** 2) - 1.0) ** 2, gpe.make_potential(gpe.GPE_POT_ELLIPSOID_SHELL, w, a, a, a)
    box = gpe.make_box(n, n, n, h, h, h, x[0], x[0], x[0])
    for target in (3.0, 1e4):
        got = gpe.gpe_tf_mu_analytic(box, pot, target * h ** 3, 1.0)
        assert abs(got - root(V, target)) <= 1e-11 * root(V, target)


def test_a_cutoff_that_is_not_a_number_selects_nothing():
    V = potential((17, 18, 19), "shell")
    box = gpe.make_box(19, 18, 17, 0.1)
    pot = gpe.make_potential(gpe.GPE_POT_HARMONIC, 1.0, 1.0, 1.0)
    for make in (lambda: gpe.gpe_grid_create_dense(box, V, np.nan),
                 lambda: gpe.gpe_grid_create_dense(box, V.astype(np.float32), np.nan),
                 lambda: gpe.gpe_grid_create_analytic(box, pot, np.nan)):
        with pytest.raises(gpe.GpeError):
            make()
