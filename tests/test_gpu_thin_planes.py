"""Planes of fewer than four rows have the stage kernel's tiles along z instead of y (thin_tiles in
csrc/common.cuh).  The same data with the rows repeated until the tiles run along y again has the same stencils
at every point, so both forms are bitwise the same, whatever the launch: the right-hand side, plane ranges of a
stage, RK4 steps, a step from host memory, a batch.  Right-hand sides also against the oracle (test_gpu_parity's 1e-12)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPES = [((20, 1, 9), None), ((17, 2, 8), 19), ((5, 3, 41), None), ((33, 3, 4), 35), ((1, 1, 30), None), ((16, 1, 2), None)]


@pytest.mark.parametrize("unequal", [False, True])
@pytest.mark.parametrize("fluid,scalar", [(0, 0), (1, 1)])
@pytest.mark.parametrize("n,pitch", SHAPES)
def test_thin_planes_equal_repeated_rows(O, n, pitch, fluid, scalar, unequal):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.batch import BatchScan
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    h = (0.5, 0.4, 0.625) if unequal else 0.5
    kw = dict(fluid=fluid, scalar=scalar, eta=1.3, ko_sigma=0.2, H0=0.3 * fluid)
    p = C.make_params(**kw)
    rng = np.random.default_rng(11 + n[0])
    data = inputs.smooth_state((1, 1, 1), seed=1, fluid=fluid, scalar=scalar, scale=0.0) + np.zeros((1, n[2], n[1], n[0]))
    data = data + rng.uniform(-0.02, 0.02, data.shape)
    reps = -(-4 // n[1]) if n[2] > 1 else 1
    dt = 0.01

    def all_calls(r):
        ev = Evolution(C.make_grid((n[0], n[1] * r, n[2]), h, pitch=pitch), p)
        ev.set_state(np.tile(data, (1, 1, r, 1)))
        start, out = ev.state.clone(), [ev.get(ev.rhs(0.2))]
        nxt, acc = torch.zeros_like(start), torch.zeros_like(start)
        cuts = sorted({0, 1, n[2] // 2, n[2]})
        for lo, hi in zip(cuts, cuts[1:]):
            C.check(C.cosmos_rk4_stage_slab(ev.g, p, 1, start, start, nxt, acc, 0.2, dt, lo, hi - lo, None, ev.ws_rhs))
        out += [ev.get(nxt), ev.get(acc)]
        ev.step(0.2, dt, 2)
        out.append(ev.get())
        b = BatchScan([ev.g, C.make_grid((8, 8, 8), 0.5), ev.g], p, [dt, dt, dt], [0.2, 0.2, 0.2], max_steps=2)
        for i in (0, 2):
            b.states[i].copy_(start)
        b.states[1].copy_(torch.from_numpy(inputs.smooth_state(8, seed=5, fluid=fluid, scalar=scalar)).reshape(-1))
        b.run(0, 2, use_graph=False)
        out += [ev.get(b.states[0]), ev.get(b.states[2])]
        host = start.cpu().pin_memory()
        C.check(C.cosmos_evolve_host(ev.g, p, host, host, torch.zeros_like(start), 2, 0.2, dt, ev.ws_rk4))
        out.append(ev.get(host))
        return out

    thin, thick = all_calls(1), all_calls(reps)
    for a, b in zip(thin, thick):
        assert np.isfinite(a).all()
        for r in range(reps):
            assert np.array_equal(a, b[:, :, r * n[1]:(r + 1) * n[1]])
    for q in (4, 5, 6):
        assert np.array_equal(thin[q], thin[3])
    ref = O.rhs(O.OGrid(n, h), O.params_array(w=p.w, t0=p.t0, slicing=p.slicing, shift=p.shift, **kw), data, 0.2)
    top = np.abs(ref).max()
    for f in range(ref.shape[0]):
        bound = 1e-12 * max(np.abs(ref[f]).max(), 1e-12 * top)
        if fluid and 24 <= f < 28:
            bound += 64 * np.finfo(float).eps * np.abs(data[24]).max() / np.min(h)
        assert np.abs(thin[0][f] - ref[f]).max() <= bound, f
