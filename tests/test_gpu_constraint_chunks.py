"""cosmos_constraints takes its finite differences a chunk of planes at a time (about 2^21 points); here
several chunks with a short last one, rows with padding, against cosmos_constraints_noalloc, which forms
them in FP64 point by point.  Noise on a flat base, spacing 1/2: the differences are as large as the
values, so both sides agree to a few roundings (1e-12 of each field's largest value)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scalar,n,pitch", [(0, (509, 512, 19), 512), (1, (256, 300, 61), 256)])
def test_chunks_equal_the_pointwise_kernel(scalar, n, pitch):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    p = C.make_params(scalar=scalar)
    ev = Evolution(C.make_grid(n, 0.5, pitch=pitch), p)
    rng = torch.Generator(device="cuda").manual_seed(4)
    base = inputs.smooth_state((1, 1, 1), seed=1, scalar=scalar, scale=0.0).reshape(-1)
    v = ev.view()
    for f, b in enumerate(base):
        v[f].uniform_(-0.05, 0.05, generator=rng).add_(float(b))
    want = torch.zeros(4 * ev.fs, dtype=torch.float64, device="cuda")
    norms = (ctypes.c_double * 8)()
    C.check(C.cosmos_constraints_noalloc(ev.g, ev.p, ev.state, want, norms))
    got, got_norms = ev.constraints(want_fields=True)
    want = ev.view(want)[..., : n[0]].cpu().numpy()
    for m in range(4):
        assert np.abs(got[m] - want[m]).max() <= 1e-12 * np.abs(want[m]).max()
    np.testing.assert_allclose(got_norms, np.array(list(norms)), rtol=1e-12)
