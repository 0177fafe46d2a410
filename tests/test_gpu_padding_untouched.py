"""Padding columns of a state are never read or written: whatever stands in them, every buffer a call fills, its
workspace included, comes out the same to the bit, and they keep what they held."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fluid,scalar", [(0, 0), (1, 1)])
@pytest.mark.parametrize("n,pitch", [((20, 12, 9), 23), ((1, 5, 3), 7), ((37, 30, 11), 300)])
def test_nothing_depends_on_the_padding(n, pitch, fluid, scalar):
    from paper_2606_02053_gb300 import build, cosmos as C, inputs
    from paper_2606_02053_gb300.batch import BatchScan

    build.build()
    g = C.make_grid(n, 0.05, pitch=pitch)
    p = C.make_params(fluid=fluid, scalar=scalar, eta=1.3, ko_sigma=0.2)
    nf, fs = C.cosmos_nfields(p), C.cosmos_field_stride(g)
    data = inputs.smooth_state(n, seed=3, fluid=fluid, scalar=scalar)
    cot = np.random.default_rng(1).uniform(-1.0, 1.0, data.shape)

    def buffer(fill, values):
        b = torch.full((nf, n[2], n[1], pitch), fill, dtype=torch.float64, device="cuda")
        b[..., : n[0]] = torch.from_numpy(values).cuda()
        return b

    def zeros(bytes_):
        return torch.zeros((bytes_ + 7) // 8, dtype=torch.float64, device="cuda")

    def run(fill):
        u, w = buffer(fill, data), buffer(fill, cot)
        out = [torch.zeros(nf * fs, dtype=torch.float64, device="cuda") for _ in range(2)]
        ws = [zeros(C.cosmos_workspace_bytes(g, p, op)) for op in (C.COSMOS_OP_RHS, C.COSMOS_OP_RK4)]
        ws.append(zeros(C.cosmos_adjoint_workspace_bytes(g, p, C.COSMOS_OP_VJP)))
        C.check(C.cosmos_rhs(g, p, u, out[0], 0.1, ws[0]))
        C.check(C.cosmos_rhs_vjp(g, p, u, w, out[1], 0.1, ws[2]))
        C.check(C.cosmos_rk4_step(g, p, u, 0.1, 0.01, ws[1]))
        scan = BatchScan([g], p, [0.01])
        scan.states[0].copy_(buffer(fill, data).reshape(-1))
        scan.run(0, 1, use_graph=False)
        torch.cuda.synchronize()
        states = [u, w, scan.states[0].view(nf, n[2], n[1], pitch)]
        pad = torch.tensor([fill], dtype=torch.float64, device="cuda").view(torch.int64)
        for s in states:
            assert (s[..., n[0] :].contiguous().view(torch.int64) == pad).all()
        return [b.view(torch.int64).clone() for b in out + ws + [s[..., : n[0]].contiguous() for s in states]]

    for a, b in zip(run(0.0), run(float("nan"))):
        assert torch.equal(a, b)
    for a, b in zip(run(1e300), run(float("inf"))):
        assert torch.equal(a, b)
