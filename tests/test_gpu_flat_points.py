"""Fluid and reverse-mode kernels over runs of points against tiles of a plane (point_launch in csrc/common.cuh).

32 x 4 tiles cover a plane of 32 x 4 points exactly; planes of other row counts are taken as runs of 128 points
of the whole grid.  On data that do not vary along y every point's result has the same operands and the same
order of operations in both, so the right-hand side and its reverse are bitwise the same, row by row.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fluid,scalar", [(0, 0), (1, 1)])
@pytest.mark.parametrize("nz", [1, 6])
def test_rhs_and_vjp_do_not_depend_on_the_launch_form(nz, fluid, scalar):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    p = C.make_params(fluid=fluid, scalar=scalar, eta=1.3, ko_sigma=0.2)
    base = inputs.smooth_state((32, 1, nz), seed=4, fluid=fluid, scalar=scalar)
    cot = np.random.default_rng(3).uniform(-1.0, 1.0, base.shape)

    def both(rows):
        g = C.make_grid((32, rows, nz), 1.0 / 32)
        ev = Evolution(g, p)
        state = np.ascontiguousarray(np.repeat(base, rows, axis=2))
        ev.set_state(state)
        w = torch.from_numpy(np.ascontiguousarray(np.repeat(cot, rows, axis=2))).cuda().reshape(-1)
        v = torch.empty_like(w)
        nb = C.cosmos_adjoint_workspace_bytes(g, p, C.COSMOS_OP_VJP)
        C.check(C.cosmos_rhs_vjp(g, p, ev.state, w, v, 0.1, torch.empty((nb + 7) // 8, dtype=torch.float64, device="cuda")))
        return ev.get(ev.rhs(0.1)), v.cpu().numpy().reshape(state.shape)

    exact = both(4)
    for rows in (1, 5, 7, 9):
        for got, ref in zip(both(rows), exact):
            for row in range(rows):
                assert np.array_equal(got[:, :, row], ref[:, :, 0]), (rows, row)
