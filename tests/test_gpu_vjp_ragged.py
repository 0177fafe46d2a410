"""The reverse kernels take runs of 32 points of the whole grid: grids whose runs cross rows and planes and end
short, with padded rows and three different spacings, against the oracle's tape.  Tolerance as in
test_gpu_adjoint: 1e-10 of each field's largest cotangent."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPES = [((9, 8, 7), 12), ((33, 5, 3), 40), ((5, 3, 2), None), ((31, 1, 4), 32), ((32, 2, 3), 33), ((1, 1, 1), 4)]


@pytest.mark.parametrize("fluid,scalar", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("n,pitch", SHAPES)
def test_vjp_on_ragged_padded_grids(O, n, pitch, fluid, scalar):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    h = (0.11, 0.08, 0.14)
    kw = dict(slicing=0, shift=1, eta=1.3, ko_sigma=0.2, fluid=fluid, scalar=scalar, H0=2.0 * fluid)
    p, g = C.make_params(**kw), C.make_grid(n, h, pitch=pitch)
    U = inputs.smooth_state(n, seed=60 + fluid + 2 * scalar, fluid=fluid, scalar=scalar, scale=0.5)
    w = np.random.default_rng(7).standard_normal(U.shape)
    ev, ew = Evolution(g, p), Evolution(g, p)
    ev.set_state(U)
    ew.set_state(w)
    v = torch.empty_like(ev.state)
    nb = C.cosmos_adjoint_workspace_bytes(g, p, C.COSMOS_OP_VJP)
    C.check(C.cosmos_rhs_vjp(g, p, ev.state, ew.state, v, 0.1, torch.empty((nb + 7) // 8, dtype=torch.float64, device="cuda")))
    ref = O.rhs_vjp(O.OGrid(n, h), O.params_array(**kw), U, w, 0.1)
    got = ev.get(v)
    top = np.abs(ref).max()
    for f in range(ref.shape[0]):
        assert np.abs(got[f] - ref[f]).max() <= 1e-10 * max(np.abs(ref[f]).max(), 1e-12 * top), f
