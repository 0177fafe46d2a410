"""The stage kernel (csrc/stage_split.cuh) against the oracle where its tiles can go wrong.

Tiles are 16 x 8 points of one plane with 3-point halos, one block works through several: grids of one
point, one below and one above a tile edge, one plane to several, more tiles than SMs, padded rows, equal
and unequal spacing, every matter variant.  The data are noise on a flat base: neighbouring values differ
by as much as they can, so the first and mixed differences pass the range of one 64-bit word and the
shortened form of the rounding runs beside the plain one.  Tolerance as in test_gpu_parity: per field
1e-12 of its largest right-hand side; noise makes the second differences the largest terms, and both sides
form them from exact neighbour differences or exactly.  The fluid's right-hand side is a difference of face
fluxes of the size of tau over h, whose own rounding (64 eps max|tau| / h) is added to its bound.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPES = [((1, 1, 1), None), ((15, 7, 3), 16), ((16, 8, 1), None), ((17, 9, 2), None), ((33, 1, 7), 35),
          ((2, 25, 5), None), ((48, 40, 12), None)]


@pytest.mark.parametrize("unequal", [False, True])
@pytest.mark.parametrize("fluid,scalar", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("n,pitch", SHAPES)
def test_rhs_of_noise_at_tile_edges(O, n, pitch, fluid, scalar, unequal):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    h = (0.5, 0.4, 0.625) if unequal else 0.5
    p = C.make_params(slicing=unequal, shift=not unequal or fluid, fluid=fluid, scalar=scalar, eta=1.3, ko_sigma=0.2,
                      H0=0.3 * fluid)
    rng = np.random.default_rng(11 + n[0])
    s = inputs.smooth_state((1, 1, 1), seed=1, fluid=fluid, scalar=scalar, scale=0.0) + np.zeros((1, n[2], n[1], n[0]))
    s = s + rng.uniform(-0.05, 0.05, s.shape)
    ev = Evolution(C.make_grid(n, h, pitch=pitch), p)
    ev.set_state(s)
    got = ev.get(ev.rhs(0.2))
    ref = O.rhs(O.OGrid(n, h), O.params_array(slicing=p.slicing, shift=p.shift, eta=p.eta, ko_sigma=p.ko_sigma, w=p.w,
                                              fluid=p.fluid, scalar=p.scalar, H0=p.H0, t0=p.t0), s, 0.2)
    top = np.abs(ref).max()
    for f in range(ref.shape[0]):
        bound = 1e-12 * max(np.abs(ref[f]).max(), 1e-12 * top)
        if fluid and 24 <= f < 28:
            bound += 64 * np.finfo(float).eps * np.abs(s[24]).max() / np.min(h)
        assert np.abs(got[f] - ref[f]).max() <= bound, (f, np.abs(got[f] - ref[f]).max(), bound)
