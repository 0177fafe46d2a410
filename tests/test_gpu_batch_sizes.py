"""The limb copy of a batch has as many blocks for every instance as the largest needs, up to 128, and repeats beyond:
batches of grids of a few points, at and past one block, and beside one whose copy repeats, bitwise against
the single-grid steps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(1, 1, 1), (4, 4, 4), (16, 1, 1)], [(16, 8, 8), (1025, 1, 1), (3, 2, 5)],
                                   [(4, 4, 4), (64, 64, 33), (9, 5, 3)]])
@pytest.mark.parametrize("fluid", [0, 1])
def test_instances_of_very_different_sizes(sizes, fluid):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.batch import BatchScan
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    p = C.make_params(fluid=fluid, eta=1.3, ko_sigma=0.2)
    grids = [C.make_grid(n, 0.05) for n in sizes]
    b = BatchScan(grids, p, [0.01] * len(grids))
    want = []
    for i, (g, n) in enumerate(zip(grids, sizes)):
        ev = Evolution(g, p)
        ev.set_state(inputs.smooth_state(n, seed=3 + i, fluid=fluid))
        b.states[i].copy_(ev.state)
        ev.step(0.0, 0.01, 1)
        want.append(ev.state)
    b.run(0, 1, use_graph=False)
    torch.cuda.synchronize()
    for got, ref in zip(b.states, want):
        assert np.isfinite(ref.cpu().numpy()).all()
        assert torch.equal(got, ref)
