"""A batch of grids with equal and with unequal spacing advances each as cosmos_rk4_step does, bitwise.

The dissipation of a grid with equal spacing is one exact integer sum, of another one a sum per axis, so the
two round differently and every instance has to take the form of its own grid, whatever the others are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

EQ, UN = 1.0 / 16, (1.0 / 16, 0.07, 0.05)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("fluid,scalar", [(0, 0), (1, 1)])
@pytest.mark.parametrize("spacings", [(EQ, UN, EQ), (UN, EQ), (EQ, EQ), (UN, UN)])
def test_mixed_spacing_equals_the_single_grid_steps(spacings, fluid, scalar, graph):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.batch import BatchScan
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    p = C.make_params(fluid=fluid, scalar=scalar, eta=1.3, ko_sigma=0.2)
    sizes = [(18, 9, 11), (17, 16, 5), (33, 8, 7)][: len(spacings)]
    grids = [C.make_grid(n, h) for n, h in zip(sizes, spacings)]
    dts = [0.01, 0.008, 0.012][: len(grids)]
    b = BatchScan(grids, p, dts, max_steps=2)
    want = []
    for i, (g, n, dt) in enumerate(zip(grids, sizes, dts)):
        s = inputs.smooth_state(n, seed=3 + i, fluid=fluid, scalar=scalar)
        ev = Evolution(g, p)
        ev.set_state(s)
        b.states[i].copy_(ev.state)
        ev.step(0.0, dt, 2)
        want.append(ev.state.clone())
    b.run(0, 2, use_graph=graph, stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    for got, ref in zip(b.states, want):
        assert np.isfinite(ref.cpu().numpy()).all()
        assert torch.equal(got, ref)
