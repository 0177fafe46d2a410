"""Host-side checks of the two-phase form of the right-hand side (codegen/bssn.py, split_layout; no GPU).

Its graph, fed with slots made from the plain inputs in the units that the layout states, gives the plain
right-hand side with the dissipation terms added; and the emitted statements, the first phase run on
region A alone and the second on region B alone, give what the graph gives.
"""
import math
import re

import numpy as np
import pytest

from paper_2606_02053_gb300.codegen import bssn
from paper_2606_02053_gb300.codegen.expr import emit_split, evaluate

VARIANTS = [(False, False), (True, False), (False, True), (True, True)]
LEN, KO, KREF = 0.37, 0.021, -0.4  # unit of length, sigma / 64 per axis sum, background trace
PLAIN = dict(eta=1.5, Kref=KREF, lapse_c1=2.0, lapse_c2=0.3, shift_on=1.0, w=1.0 / 3.0)
SPLIT = dict(eta=1.5 * LEN ** 2, lapse_c1=2.0 * LEN, lapse_c2=0.3 * LEN, shift_on=1.0, w=1.0 / 3.0, len=LEN,
             c75=0.75 * LEN, c43=4.0 / 3.0 * LEN)


def degree(f, fluid, scalar):
    """Inverse lengths that field f carries."""
    if f >= 24:
        return 2 if fluid and f < 28 else int(f == 25 + 4 * fluid)
    return int(7 <= f <= 16 or f >= 21)


def plain_inputs(fluid, scalar, rng):
    L = bssn.layout(fluid, scalar)
    v = {nm: 0.2 * rng.standard_normal() for nm in L["names"]}
    v.update({k: x + 0.05 * rng.standard_normal() for k, x in
              dict(u0=1.0, u1=1.2, u4=1.1, u6=0.9, u17=1.0, u24=2.0, rho=1.1).items() if k in v})
    v.update({f"k{f}": rng.standard_normal() for f in range(L["nf"])})  # Kreiss-Oliger brackets
    return L, v


def slots(L, v, fluid, scalar):
    """The split form's inputs: differences in units of l without their field's l."""
    out = {}
    for f in range(L["nf"]):
        d = 0 if 21 <= f < 24 else degree(f, fluid, scalar)
        out[f"u{f}"] = v[f"u{f}"] * LEN ** d
        if f in L["d1"]:
            for k in range(3):
                out[f"d{f}_{k}"] = v[f"d{f}_{k}"] * LEN
            adv = sum(v[f"u{18 + k}"] * out[f"d{f}_{k}"] for k in range(3))
            out[f"m{f}"] = LEN ** degree(f, fluid, scalar) * (KO * v[f"k{f}"] + adv)
        if f in L["d2"]:
            for p in range(6):
                out[f"dd{f}_{p}"] = v[f"dd{f}_{p}"] * LEN ** 2
    out["kdiff"] = v["u7"] - KREF
    out["ichi"] = 1.0 / v["u0"]
    gt = np.array([[v["u1"], v["u2"], v["u3"]], [v["u2"], v["u4"], v["u5"]], [v["u3"], v["u5"], v["u6"]]])
    for m, (a, b) in enumerate([(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]):
        out[f"gu{m}"] = np.linalg.inv(gt)[a, b]
    if fluid:
        out["rho"] = v["rho"] * LEN ** 2
    return out


@pytest.mark.parametrize("fluid,scalar", VARIANTS)
def test_split_form_is_the_plain_right_hand_side(fluid, scalar):
    rng = np.random.default_rng(5 + 2 * fluid + scalar)
    gp, _, plain = bssn.algebra(fluid, scalar)
    gs, S, split = bssn.algebra(fluid, scalar, split=True)
    for _ in range(5):
        L, v = plain_inputs(fluid, scalar, rng)
        want = np.array(evaluate(gp, plain, v, PLAIN), dtype=float)
        for f in range(L["nf"]):
            if not (fluid and 24 <= f < 28):
                want[f] += KO / LEN * v[f"k{f}"]
        got = np.array(evaluate(gs, split, slots(L, v, fluid, scalar), SPLIT), dtype=float)
        got *= [LEN ** -(degree(f, fluid, scalar) + 1) for f in range(L["nf"])]
        assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    # every output has a slot of its own in region B, read by that output alone or by none
    assert len(set(S["out"])) == L["nf"]


@pytest.mark.parametrize("fluid,scalar", VARIANTS)
def test_emitted_phases_read_their_own_region(fluid, scalar):
    rng = np.random.default_rng(9)
    g, S, out = bssn.algebra(fluid, scalar, split=True)
    src = emit_split(g, "f", S["a"], S["b"], out, g.cut, "P")
    L, v = plain_inputs(fluid, scalar, rng)
    val = slots(L, v, fluid, scalar)
    want = np.array(evaluate(g, out, val, SPLIT), dtype=float)
    env = {"ina": [val[nm] for nm in S["a"]], "p": type("P", (), SPLIT), "sqrt": math.sqrt,
           "k": type("K", (), dict(nz=-0.0, one=1.0, two=2.0, half=0.5)), "fma": lambda a, b, c: a * b + c}
    got = np.full(len(out), np.nan)
    body = src[src.index("{") + 1:src.rindex("}")]
    for line in body.split("\n"):
        line = line.strip()
        if line == "next();":  # region A is gone from here on
            env.pop("ina")
            env["inb"] = [val.get(nm, np.nan) for nm in S["b"]]
        elif m := re.fullmatch(r"const double (\w+) = (.+);", line):
            env[m.group(1)] = eval(m.group(2), env)
        elif m := re.fullmatch(r"out\[(\d+)\] = (\w+);", line):
            got[int(m.group(1))] = env[m.group(2)]
    assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
