"""The calls that launch the stage kernel, whose offsets within a field are 32-bit counts of bytes, refuse a field
of more than 2^29 points before anything else; at 2^29 they go on to the workspace, here too small."""
import ctypes

import pytest


def calls(C, n):
    L = C.lib()
    g, p = ctypes.byref(C.make_grid(n, 0.05)), ctypes.byref(C.make_params())
    u = [ctypes.c_void_p((q + 1) << 12) for q in range(5)]  # never dereferenced
    host = (ctypes.c_void_p * 1)(1 << 40)
    out = (ctypes.c_void_p * 1)(1 << 45)
    dev = (ctypes.c_void_p * 1)(1 << 12)
    ws = ctypes.c_void_p(1 << 20)
    return {
        "rhs": lambda: L.cosmos_rhs(g, p, u[0], u[1], 0.0, ws, 0, None),
        "stage": lambda: L.cosmos_rk4_stage(g, p, 1, u[0], u[0], u[1], u[2], 0.0, 0.1, ws, 0, None),
        "slab": lambda: L.cosmos_rk4_stage_slab(g, p, 1, u[0], u[0], u[1], u[2], 0.0, 0.1, 0, 1, None, ws, 0, None),
        "pass": lambda: L.cosmos_stage_pass(g, p, 2, 1, u[0], u[0], u[1], u[2], 0.0, 0.1, ws, 0, None),
        "step": lambda: L.cosmos_rk4_step(g, p, u[0], 0.0, 0.1, ws, 0, None),
        "step_stages": lambda: L.cosmos_rk4_step_stages(g, p, u[0], 0.0, 0.1, u[1], u[2], u[3], ws, 0, None),
        "host": lambda: L.cosmos_evolve_host(g, p, host[0], out[0], u[0], 1, 0.0, 0.1, ws, 0, None),
        "many": lambda: L.cosmos_evolve_host_many(g, p, 1, host, out, dev, 1, 1, 0.0, 0.1, ws, 0, None),
        "adjoint": lambda: L.cosmos_adjoint_step(g, p, u[0], u[1], u[2], 0.0, 0.1, ws, 0, None),
    }


@pytest.mark.parametrize("name", ["rhs", "stage", "slab", "pass", "step", "step_stages", "host", "many", "adjoint"])
def test_fields_beyond_32_bit_byte_offsets_are_refused(name):
    from paper_2606_02053_gb300 import build, cosmos as C

    build.build()
    assert calls(C, (1024, 1024, 512))[name]() == C.COSMOS_EWORKSPACE
    assert calls(C, (1024, 1024, 513))[name]() == C.COSMOS_EINVAL


def test_batches_refuse_such_a_field():
    from paper_2606_02053_gb300 import build, cosmos as C

    build.build()
    for nz, ok in ((512, True), (513, False)):
        grids = [C.make_grid((16, 16, 16), 0.05), C.make_grid((1024, 1024, nz), 0.05)]
        assert (C.cosmos_batch_workspace_bytes(grids, C.make_params(), 1) > 0) == ok


def test_a_refined_step_refuses_such_a_level():
    from paper_2606_02053_gb300 import build, cosmos as C

    build.build()
    L, p = C.lib(), C.make_params()
    for nz, code in ((512, C.COSMOS_EWORKSPACE), (513, C.COSMOS_EINVAL)):
        m = C.cosmos_fmr()
        m.levels = 1
        m.grid[0] = C.make_grid((1024, 1024, nz), 0.05)
        need = L.cosmos_fmr_workspace_bytes(ctypes.byref(m), ctypes.byref(p))
        states = (ctypes.c_void_p * 1)(1 << 12)
        ws = ctypes.c_void_p(1 << 20)
        got = L.cosmos_fmr_step(ctypes.byref(m), ctypes.byref(p), states, 0.0, 0.1, ws, 0, None)
        assert need > 0 and got == code
