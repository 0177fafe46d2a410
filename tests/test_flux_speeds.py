"""The Kurganov-Tadmor flux of the generated code (codegen/fluid.py) against the scheme written out: the dissipation
takes the largest modulus of the characteristic speeds alpha v^d (1 - w) / (1 - w v^2) +- .. - beta^d of both
sides, whatever the sign of the lapse.  Both are plain FP64 evaluations of some 200 operations without
cancellation beyond the sums of the two sides: 1e-13 of the largest flux."""
import math

import numpy as np
import pytest

from paper_2606_02053_gb300.codegen import fluid
from paper_2606_02053_gb300.codegen.expr import evaluate

SYM = [[0, 1, 2], [1, 3, 4], [2, 4, 5]]


def minmod(a, b):
    return 0.0 if a * b <= 0 else (a if abs(a) <= abs(b) else b)


def textbook(v, d, w):
    """H_tau, H_S0, H_S1, H_S2 through one face along axis d."""
    q = np.array([[v[f"q{o}_{m}"] for m in range(4)] for o in range(4)])
    left = [q[1][m] + 0.5 * minmod(q[1][m] - q[0][m], q[2][m] - q[1][m]) for m in range(4)]
    right = [q[2][m] - 0.5 * minmod(q[2][m] - q[1][m], q[3][m] - q[2][m]) for m in range(4)]
    mean = {k: 0.5 * (v[k + "0"] + v[k + "1"]) for k in ("chi", "alpha", "beta")}
    gt = np.array([0.5 * (v[f"gt0_{m}"] + v[f"gt1_{m}"]) for m in range(6)])[SYM]
    up = mean["chi"] * np.linalg.inv(gt)
    U, F, speeds = [], [], []
    for side in (left, right):
        rho, vl = side[0], np.array(side[1:])
        vu = up @ vl
        v2 = vu @ vl
        W2, P = 1 / (1 - v2), w * rho
        E, J = (rho + P) * W2 - P, (rho + P) * W2 * vl
        U.append(np.array([E, *J]))
        flux = mean["alpha"] * (rho + P) * W2 * vu[d] * np.array([1.0, *vl])
        flux[1 + d] += mean["alpha"] * P
        F.append(flux - mean["beta"] * U[-1])
        root = math.sqrt(w * (1 - v2) * (up[d, d] * (1 - v2 * w) - vu[d] ** 2 * (1 - w)))
        speeds += [abs(mean["alpha"] / (1 - v2 * w) * (vu[d] * (1 - w) + s * root) - mean["beta"]) for s in (1, -1)]
    return 0.5 * mean["chi"] ** -1.5 * (F[0] + F[1] - max(speeds) * (U[1] - U[0]))


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("d", [0, 1, 2])
def test_flux_equals_the_scheme_for_either_sign_of_the_lapse(d, sign):
    g, names, out = fluid.face_flux(d)
    rng = np.random.default_rng(5 + d)
    w = 0.3
    for _ in range(50):
        v = {}
        for o in range(4):
            v[f"q{o}_0"] = rng.uniform(0.5, 1.0)
            v.update({f"q{o}_{m}": rng.uniform(-0.3, 0.3) for m in (1, 2, 3)})
        for s in range(2):
            v[f"chi{s}"], v[f"alpha{s}"], v[f"beta{s}"] = rng.uniform(0.8, 1.2), sign * rng.uniform(0.4, 1.0), rng.uniform(-0.4, 0.4)
            for m, base in enumerate((1, 0, 0, 1, 0, 1)):
                v[f"gt{s}_{m}"] = base + rng.uniform(-0.05, 0.05)
        got = np.array(evaluate(g, out, v, dict(w=w, sqrt_w=math.sqrt(w))), dtype=float)
        want = textbook(v, d, w)
        assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
