"""cosmos_constraints asks for its partial sums and, with the fluid, the primitives, on every grid: 8 doubles per
block of 32 x 4 points of a plane (half a byte a point where the tiles are full) and 4 doubles a point."""
import pytest


@pytest.mark.parametrize("n", [(256, 256, 256), (2048, 2048, 32), (4096, 4096, 8), (8192, 4096, 4), (32, 4, 1)])
@pytest.mark.parametrize("fluid", [0, 1])
def test_workspace_is_the_partial_sums(n, fluid):
    from paper_2606_02053_gb300 import build, cosmos as C

    build.build()
    g, p = C.make_grid(n, 1.0 / n[0]), C.make_params(fluid=fluid)
    points = n[0] * n[1] * n[2]
    assert C.cosmos_workspace_bytes(g, p, C.COSMOS_OP_CONSTRAINTS) <= points // 2 + 32 * points * fluid + 4096
