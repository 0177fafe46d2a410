"""The inverse metric and 1/chi that the limb copy forms (csrc/limbs.cu), through the right-hand side.

The copy takes blocks of 256 points of chi and the metric and of 1024 points of each other field: grids of
one point, of one below, at and one above those edges, and of several, with and without padded rows, on a
metric that is far from flat at every point.  Tolerance as in test_gpu_parity: per field 1e-12 of its
largest right-hand side (an FP64 sum of some thousand rounded terms, the noise making the differences the
largest of them, on a metric of condition below 4).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPES = [((1, 1, 1), None), ((255, 1, 1), None), ((16, 8, 2), None), ((257, 1, 1), None), ((11, 31, 3), None),
          ((16, 8, 8), None), ((25, 41, 1), None), ((30, 20, 9), 37)]


@pytest.mark.parametrize("n,pitch", SHAPES)
def test_rhs_on_a_curved_metric_at_block_edges(O, n, pitch):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    rng = np.random.default_rng(5 + n[0])
    s = inputs.smooth_state((1, 1, 1), seed=2, scale=0.0) + np.zeros((1, n[2], n[1], n[0]))
    s = s + rng.uniform(-0.05, 0.05, s.shape)
    s[0] = rng.uniform(0.5, 2.0, s[0].shape)           # chi
    s[1:7] += rng.uniform(-0.15, 0.15, s[1:7].shape)   # the conformal metric, diagonally dominant
    ev = Evolution(C.make_grid(n, 0.5, pitch=pitch), C.make_params(eta=1.3, ko_sigma=0.2))
    ev.set_state(s)
    got = ev.get(ev.rhs(0.2))
    ref = O.rhs(O.OGrid(n, 0.5), O.params_array(eta=1.3, ko_sigma=0.2), s, 0.2)
    top = np.abs(ref).max()
    for f in range(ref.shape[0]):
        bound = 1e-12 * max(np.abs(ref[f]).max(), 1e-12 * top)
        assert np.abs(got[f] - ref[f]).max() <= bound, (f, np.abs(got[f] - ref[f]).max(), bound)
