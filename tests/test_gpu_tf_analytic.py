"""Thomas-Fermi mu of analytic potentials on boxes around the kernel's runs of
128 cells and their parts of 32: against the root found by sorting the cells'
values.  Few cells below mu, some, and every one."""
import numpy as np
import pytest

from paper_2603_05447_gb300 import gpe
from test_gpu_tf import root

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [1, 31, 32, 33, 127, 128, 129, 161, 300])
@pytest.mark.parametrize("kind", ["harmonic", "shell"])
@pytest.mark.parametrize("offset", [0.0, 7.3])
def test_tf_mu_analytic_is_the_root(nx, kind, offset):
    ny, nz, h = 21, 18, 0.02
    axes = [(np.arange(n) - (n - 1) / 2) * h for n in (nx, ny, nz)]
    axes[0] = axes[0] + offset          # the trap's centre is far outside the box
    x, y, z = axes[0], axes[1][:, None], axes[2][:, None, None]
    if kind == "harmonic":
        w = (3.0, 2.5, 4.0)
        V = 0.5 * ((w[0] * x) ** 2 + (w[1] * y) ** 2 + (w[2] * z) ** 2)
        pot = gpe.make_potential(gpe.GPE_POT_HARMONIC, *w)
    else:
        w, a = 40.0, (0.16 + offset, 0.15, 0.14)
        V = 0.5 * w * w * (np.sqrt((x / a[0]) ** 2 + (y / a[1]) ** 2 + (z / a[2]) ** 2) - 1.0) ** 2
        pot = gpe.make_potential(gpe.GPE_POT_ELLIPSOID_SHELL, w, *a)
    box = gpe.make_box(nx, ny, nz, h, h, h, *(float(v[0]) for v in axes))
    for target in (1e-3, 30.0, 1e3 * V.size):
        got, want = gpe.gpe_tf_mu_analytic(box, pot, target * h ** 3, 1.0), root(V, target)
        # FP64 sums of up to 1e5 terms; the cells' values differ by a few roundings
        assert abs(got - want) <= 1e-11 * max(abs(want), 1.0)


@pytest.mark.parametrize("kind,w,h", [("harmonic", 4.58e-23, 1e13), ("harmonic", 4.7e-23, 1e13), ("harmonic", 2e21, 2.1e-23), ("harmonic", 3e-38, 1e25),
                                      ("shell", 1e-30, 0.1), ("shell", 3e-16, 0.1)])
def test_weak_traps_and_small_boxes_lose_no_cells(kind, w, h):
    """Frequencies and coordinates whose squares FP32 cannot hold: the builder's region and
    the Thomas-Fermi mu still follow from the cells' FP64 values."""
    n = 40
    x = (np.arange(n) - (n - 1) / 2) * h
    r2 = x ** 2 + (x ** 2)[:, None] + (x ** 2)[:, None, None]
    if kind == "harmonic":
        V, pot = 0.5 * w * w * r2, gpe.make_potential(gpe.GPE_POT_HARMONIC, w, w, w)
    else:
        a = 12 * h
        V, pot = 0.5 * w * w * (np.sqrt(r2) / a - 1.0) ** 2, gpe.make_potential(gpe.GPE_POT_ELLIPSOID_SHELL, w, a, a, a)
    box = gpe.make_box(n, n, n, h)
    v = np.sort(V.ravel())
    for count in (300, 3000, 30000):
        cut = 0.5 * (v[count - 1] + v[np.searchsorted(v, v[count - 1] * 1.000001)])  # between two values
        grid = gpe.gpe_grid_create_analytic(box, pot, cut)
        assert gpe.gpe_grid_get_info(grid).n_active == int((V < cut).sum())
        gpe.gpe_grid_destroy(grid)
        target = float(np.maximum(cut - V, 0.0).sum())
        got = gpe.gpe_tf_mu_analytic(box, pot, target, h ** 3)
        assert abs(got - root(V, target)) <= 1e-11 * root(V, target)
