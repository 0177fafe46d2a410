"""A recording pass of a stage (cosmos_stage_pass, pass 2 + 32) leaves what it reads as it was: run again on
the same passes 0 and 1, it writes the same stage state and accumulator and records the same exponents."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fluid,scalar", [(0, 0), (1, 1)])
def test_a_recording_pass_can_be_repeated(fluid, scalar):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.evolve import Evolution

    build.build()
    n, dt = (24, 18, 7), 0.01
    p = C.make_params(fluid=fluid, scalar=scalar, eta=1.3, ko_sigma=0.2)
    ev = Evolution(C.make_grid(n, 1.0 / 24), p)
    s = inputs.smooth_state(n, seed=5, fluid=fluid, scalar=scalar)
    s[20] *= 1e-9  # a field whose exponent the first stage raises
    ev.set_state(s)
    un = ev.state
    A, B, acc = (torch.zeros_like(un) for _ in range(3))

    def run(q, stage, us, out):
        C.check(C.cosmos_stage_pass(ev.g, p, q, stage, us, un, out, acc, 0.0, dt, ev.ws_rhs))

    def second():
        run(0, 2, A, B)
        run(1 + 16, 2, A, B)
        run(2, 2, A, B)
        return B.clone(), acc.clone()

    for q in (0, 1, 2 + 64):
        run(q, 1, un, A)
    first = A.clone(), acc.clone()
    want = second()
    for q in (0, 1, 2 + 64, 2 + 32, 2 + 32):
        run(q, 1, un, A)
        if q >= 32:
            assert torch.equal(A, first[0]) and torch.equal(acc, first[1]), q
    for got, ref in zip(second(), want):
        assert torch.equal(got, ref)
