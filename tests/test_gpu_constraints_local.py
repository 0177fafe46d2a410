"""The constraints of a point depend on its neighbourhood only.

Small values of a field: with a flat metric and nothing but K, M^i = -2/3 d_i K.  K is a Gaussian of width
0.05 of the box without a base, so its values span 22 orders of magnitude, and the stencil
(8 (f+1 - f-1) - (f+2 - f-2)) / 12 h is a difference of two rounded differences times rounded coefficients
(4 roundings of each term) and M^i takes some 8 more multiply-adds with exact zeros: 16 u times the sum of
the terms' moduli bounds the error at each point, however small.

One NaN: outside the stencils that reach it (2 points along each axis) the fields are bitwise those without
it, and the largest moduli are taken over the values that are numbers.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def evolution(n, h):
    from paper_2606_02053_gb300 import build, cosmos as C
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    return Evolution(C.make_grid(n, h), C.make_params())


def flat(n):
    from paper_2606_02053_gb300 import inputs

    return inputs.smooth_state((1, 1, 1), seed=1, scale=0.0) * np.ones((1, n[2], n[1], n[0]))


def test_small_values_keep_their_accuracy():
    n, h = (128, 8, 5), 1.0 / 128
    s = flat(n)
    s[1:] = 0.0  # flat space: unit metric and lapse, everything else zero
    for f in (0, 1, 4, 6, 17):
        s[f] = 1.0
    x = (np.arange(n[0]) - 64) * h
    s[7] = np.exp(-0.5 * (x / 0.05) ** 2)
    ev = evolution(n, h)
    ev.set_state(s)
    got, norms = ev.constraints(want_fields=True)
    K = s[7].astype(np.longdouble)
    d = {o: np.roll(K, -o, axis=2) for o in (-2, -1, 1, 2)}
    want = -2 / np.longdouble(3) * (8 * (d[1] - d[-1]) - (d[2] - d[-2])) / (12 * np.longdouble(h))
    size = 2 / np.longdouble(3) * (8 * np.abs(d[1] - d[-1]) + np.abs(d[2] - d[-2])) / (12 * np.longdouble(h))
    assert (np.abs(got[1] - want) <= 16 * 2.0**-53 * size).all(), float((np.abs(got[1] - want) / size).max())
    assert (got[2] == 0).all() and (got[3] == 0).all()


@pytest.mark.parametrize("field", [0, 2, 7])
def test_a_nan_stays_in_its_neighbourhood(field):
    n = (37, 21, 17)
    rng = np.random.default_rng(9)
    s = flat(n) + rng.uniform(-0.02, 0.02, (24, n[2], n[1], n[0]))
    ev = evolution(n, 0.5)
    ev.set_state(s)
    clean, _ = ev.constraints(want_fields=True)
    s[field, 8, 10, 30] = np.nan
    ev.set_state(s)
    got, norms = ev.constraints(want_fields=True)
    away = np.ones(clean.shape[1:], bool)
    away[6:11, 8:13, 28:33] = False
    assert np.array_equal(got[:, away], clean[:, away])
    assert np.isnan(got[0, 8, 10, 30])
    for m in range(4):
        finite = np.abs(got[m][np.isfinite(got[m])])
        assert norms[4 + m] == finite.max()
