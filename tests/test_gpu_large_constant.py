"""A constant of any finite size has zero differences: the right-hand side of a scalar field that holds one near the
end of the FP64 range is bitwise that of one that holds 1 (its potential is zero, only its differences enter)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unequal", [False, True])
@pytest.mark.parametrize("value", [1.5 * 2.0**1022, -1.7e308, 2.0**1021, 2.0**-1000])
def test_a_constant_scalar_field_does_not_enter(value, unequal):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    n = (18, 9, 5)
    ev = Evolution(C.make_grid(n, (0.5, 0.4, 0.6) if unequal else 0.5), C.make_params(scalar=1, ko_sigma=0.2))
    s = inputs.smooth_state(n, seed=2, scalar=1)

    def rhs(phi):
        s[24] = phi
        ev.set_state(s)
        return ev.get(ev.rhs(0.0))

    want = rhs(1.0)
    assert np.isfinite(want).all()
    assert np.array_equal(rhs(value), want)
