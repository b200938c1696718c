"""Steps captured by the caller in a CUDA graph of its own: replayed, they give the
eager calls' bits, also after the state's own graph length has grown (which asks
for a longer table of the ramp's schedule)."""
import numpy as np
import pytest

from paper_2603_05447_gb300 import gpe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (18, 21, 24)


@pytest.mark.parametrize("stencil,integrator", [(7, gpe.GPE_RK4), (7, gpe.GPE_RKCK), (19, gpe.GPE_RK4)])
@pytest.mark.parametrize("blend", [False, True])
def test_replayed_steps_match_eager_ones(blend, stencil, integrator):
    rng = np.random.default_rng(8)
    V0, V1 = rng.uniform(0.0, 2.0, SHAPE), rng.uniform(0.0, 4.0, SHAPE)
    psi = (rng.normal(size=SHAPE) + 1j * rng.normal(size=SHAPE)).astype(np.complex64) / 90.0
    grid = gpe.gpe_grid_create_dense(gpe.make_box(*SHAPE[::-1], 0.5), V0, 1e9, gpe.make_opts((8, 8, 4), stencil=stencil))
    gpe.gpe_grid_set_potential(grid, 1, V1)
    a, b = (gpe.gpe_state_create(grid, gpe.GPE_C64) for _ in range(2))
    p = (gpe.real_params(0.5, 0.01, gpe.GPE_V_BLEND, [0.2, 0.9, 0.4], 0.5) if blend else gpe.real_params(0.5, 0.01))
    p.integrator = integrator
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    got = []
    try:
        for st in (a, b):
            gpe.gpe_state_load(st, psi, gpe.GPE_LAYOUT_DENSE)
            gpe.gpe_step_real(st, p, 3, stream=side)  # what is made on first use
        side.synchronize()
        with torch.cuda.graph(graph, stream=side):
            gpe.gpe_step_real(a, p, 3, 0.1, stream=side)
        gpe.gpe_state_set_graph(a, 3000)
        graph.replay()
        torch.cuda.synchronize()
        gpe.gpe_step_real(a, p, 2, 0.2, stream=side)
        gpe.gpe_step_real(b, p, 3, 0.1, stream=side)
        gpe.gpe_step_real(b, p, 2, 0.2, stream=side)
        side.synchronize()
        for st in (a, b):
            out = np.empty(SHAPE, np.complex64)
            gpe.gpe_state_store(st, out, gpe.GPE_LAYOUT_DENSE)
            got.append(out)
    finally:
        del graph
        for st in (a, b):
            gpe.gpe_state_destroy(st)
        gpe.gpe_grid_destroy(grid)
    assert np.array_equal(got[0], got[1]) and np.abs(got[0] - psi).max() > 1e-4
