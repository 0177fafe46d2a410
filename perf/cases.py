"""What a user of this framework has it do, as cases whose time and results can be taken.

A case names a call (right-hand side, RK4 steps, a batched scan, steps of a refined hierarchy, a reverse
step, a vector-Jacobian product, the constraints), the matter, the initial data and the grid.  The inputs are
made on the GPU from the seed by plain torch, the call goes through the package's public entry points, and
``exact`` evaluates the same call in plain torch in FP64.
"""
import math
import random

import torch

from paper_2606_02053_gb300 import cosmos as C
from paper_2606_02053_gb300 import inputs
from paper_2606_02053_gb300.batch import BatchScan
from paper_2606_02053_gb300.evolve import Evolution
from paper_2606_02053_gb300.fmr import Hierarchy

DEV = "cuda"
CFL = 0.25
H0 = 40.0  # background expansion rate of the collapse workloads (H0 L = 40, unit box)
MATTER = {"vac": (0, 0), "fluid": (1, 0), "scalar": (0, 1), "both": (1, 1)}
PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
SYM = [[0, 1, 2], [1, 3, 4], [2, 4, 5]]


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def _one(call, matter, data, n, name=None, **more):
    n = (n, n, n) if isinstance(n, int) else n
    c = dict(call=call, matter=matter, data=data, nx=n[0], ny=n[1], nz=n[2], pitch=n[0], steps=1, unequal=False,
             harmonic=False, frozen=False)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one right-hand side of a tiny ragged grid with a scalar field: a parity check or a driver that
        # integrates in time by itself; launches and latency are all of it
        _one("rhs", "scalar", "smooth", (20, 12, 9), "rhs scalar 20x12x9"),
        # the 32^3 gauge-wave test, all of its 20 steps
        _one("step", "vac", "gauge", 32, "gauge wave 32, 20 steps", steps=20),
        # one step of the smallest grid of a threshold scan run by itself
        _one("step", "fluid", "flrw", 64, "collapse 64"),
        # fluid and scalar on an odd-sized grid with padded rows and unequal spacing
        _one("step", "both", "smooth", (97, 80, 66), "fluid+scalar 97x80x66", pitch=104, unequal=True),
        # the 128^3 curvature-perturbation run
        _one("step", "fluid", "flrw", 128, "collapse 128"),
        # a large ragged vacuum grid on which every field varies along every axis
        _one("step", "vac", "smooth", (250, 198, 203), "vacuum 250x198x203"),
        # the headline sweep
        _one("step", "vac", "gauge", 256, "gauge wave 256"),
        # a share of the batched threshold scan: uneven grids of 64^3 to 96^3 advanced together
        _one("scan", "fluid", "flrw", 96, "scan of 16", count=16, n_lo=64, draw=2606),
        # a refined run: the periodic box and two nested boxes around its centre
        _one("fmr", "fluid", "flrw", 128, "refined 128+96+96", levels=3, n_child=96),
        # one reverse step of the gradient run, given the forward stage states
        _one("adjoint", "fluid", "smooth", 96, "reverse step 96"),
        # one vector-Jacobian product of the right-hand side of a small odd-sized vacuum grid
        _one("vjp", "vac", "smooth", (45, 33, 28), "vjp vacuum 45x33x28"),
        # the constraint fields and norms that a run reports on its way
        _one("constraints", "fluid", "smooth", 128, "constraints 128"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["rhs", "step", "step", "step", "scan", "fmr", "adjoint", "vjp", "constraints"])
    if call == "scan":
        lo = rng.randint(48, 72)
        return _one("scan", "fluid", "flrw", rng.randint(lo + 4, 96), count=rng.randint(3, 12), n_lo=lo,
                    draw=rng.randrange(1 << 20))
    if call == "fmr":
        n = rng.randint(48, 112)
        return _one("fmr", "fluid", "flrw", n, levels=rng.randint(2, 3), n_child=rng.randint(32, min(88, 2 * (n // 2 - 6))))
    matter = rng.choice(["vac", "fluid", "scalar", "both"])
    big = {"rhs": 200, "step": 200, "adjoint": 72, "vjp": 72, "constraints": 200}[call]
    n = tuple(_log_int(rng, 9, big) for _ in range(3))
    data = "smooth"
    if matter == "vac" and call != "constraints" and rng.random() < 0.3:
        data = "gauge"
    elif matter == "fluid" and call in ("rhs", "step") and rng.random() < 0.6:
        data, n = "flrw", (_log_int(rng, 32, 160),) * 3
    unequal = data == "smooth" and rng.random() < 0.3
    pitch = n[0] if rng.random() < 0.6 else n[0] + rng.randint(1, 7)
    return _one(call, matter, data, n, pitch=pitch, unequal=unequal, harmonic=rng.random() < 0.25,
                frozen=rng.random() < 0.25, steps=rng.randint(1, 3) if call == "step" and n[0] * n[1] * n[2] < 1 << 19 else 1)


# ---------------------------------------------------------------------------
# Inputs, in plain torch
# ---------------------------------------------------------------------------
def _n(case):
    return case["nx"], case["ny"], case["nz"]


def _spacing(case):
    n = _n(case)
    return tuple(1.0 / v for v in n) if case["unequal"] else (1.0 / case["nx"],) * 3


def _plain_params(case):
    fluid, scalar = MATTER[case["matter"]]
    return dict(slicing=int(case["harmonic"]), shift=int(not case["frozen"]), fluid=fluid, scalar=scalar, eta=2.0,
                ko_sigma=0.1, w=1.0 / 3.0, H0=H0 if case["data"] == "flrw" else 0.0, t0=0.0)


def _axes(n, h, x0):
    ax = [x0[d] + h[d] * torch.arange(n[d], dtype=torch.float64, device=DEV) for d in range(3)]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _smooth(n, rng, matter):
    """A base state near flat space plus three random Fourier modes per field (inputs.smooth_state's ranges)."""
    fluid, scalar = MATTER[matter]
    base = list(inputs._BASE_BSSN) + [1.0, 0.0, 0.0, 0.0] * fluid + [0.0, 0.0] * scalar
    amp = list(inputs._AMP_BSSN) + [0.2, 0.05, 0.05, 0.05] * fluid + [0.2, 0.2] * scalar
    x, y, z = _axes(n, (2.0 * math.pi / n[0], 2.0 * math.pi / n[1], 2.0 * math.pi / n[2]), (0.0, 0.0, 0.0))
    out = torch.empty((len(base), n[2], n[1], n[0]), dtype=torch.float64, device=DEV)
    for f in range(len(base)):
        out[f] = base[f]
        for _ in range(3):
            k = [rng.randint(-2, 2) for _ in range(3)]
            c, ph = 0.5 * amp[f] * rng.uniform(-1.0, 1.0), rng.uniform(0.0, 2.0 * math.pi)
            out[f] += c * torch.sin(k[0] * x + k[1] * y + k[2] * z + ph)
    return out


def _gauge_wave(n, h, rng):
    A, t = rng.uniform(0.008, 0.012), rng.uniform(0.0, 1.0)
    Lx = n[0] * h[0]
    x, _, _ = _axes(n, h, (0.0, 0.0, 0.0))
    ph = 2.0 * math.pi * (x - t) / Lx
    H, dtH = 1.0 - A * torch.sin(ph), A * (2.0 * math.pi / Lx) * torch.cos(ph)
    sH, chi = torch.sqrt(H), H ** (-1.0 / 3.0)
    Kxx = -dtH / (2.0 * sH)
    K = Kxx / H
    out = torch.zeros((24, n[2], n[1], n[0]), dtype=torch.float64, device=DEV)
    for f, v in {0: chi, 1: H ** (2.0 / 3.0), 4: chi, 6: chi, 7: K, 8: chi * (Kxx - H * K / 3.0), 11: -chi * K / 3.0,
                 13: -chi * K / 3.0, 14: -(2.0 / 3.0) * H ** (-5.0 / 3.0) * dtH, 17: sH}.items():
        out[f] = v
    return out


def _shape(rng, scan=False):
    """Amplitude, width and axis ratios of a curvature perturbation."""
    q = [rng.uniform(0.8, 1.2) for _ in range(3)] if scan else [1.0, 1.0, 1.0]
    return rng.uniform(0.45, 0.55), rng.uniform(0.11, 0.14), q


def _collapse(n, h, x0, shape):
    """FLRW + zeta at leading gradient order, the fluid at rest with its energy from the Hamiltonian constraint."""
    mu, sigma, q = shape
    x, y, z = _axes(n, h, x0)
    zeta = mu * torch.exp(-((x / q[0]) ** 2 + (y / q[1]) ** 2 + (z / q[2]) ** 2) / (2.0 * sigma * sigma))
    out = torch.zeros((28, n[2], n[1], n[0]), dtype=torch.float64, device=DEV)
    out[0] = torch.exp(-2.0 * zeta)
    out[1] = out[4] = out[6] = out[17] = 1.0
    out[7] = -3.0 * H0
    chi = out[0]
    dchi = [_d1(chi, d, h) for d in range(3)]
    lap = sum(_d2(chi, d, d, h) for d in range(3))
    R = 2.0 * lap - 2.5 * sum(v * v for v in dchi) / chi  # of the conformally flat metric delta_ij / chi
    out[24] = (R + (2.0 / 3.0) * out[7] ** 2) / (16.0 * math.pi) / (chi * torch.sqrt(chi))
    return out


def _initial(case, seed):
    rng = random.Random(seed)
    n, h = _n(case), _spacing(case)
    if case["data"] == "gauge":
        return _gauge_wave(n, h, rng)
    if case["data"] == "flrw":
        return _collapse(n, h, tuple(-(v // 2) * s for v, s in zip(n, h)), _shape(rng))
    return _smooth(n, rng, case["matter"])


def _cotangent(case, seed):
    fluid, scalar = MATTER[case["matter"]]
    g = torch.Generator(device=DEV).manual_seed(seed + 77)
    return torch.randn((24 + 4 * fluid + 2 * scalar, case["nz"], case["ny"], case["nx"]), generator=g, device=DEV,
                       dtype=torch.float64)


def _scan_grids(case):
    return [i["n"] for i in inputs.scan_instances(case["count"], case["draw"], case["n_lo"], case["nx"])]


def _scan_states(case, seed):
    rng = random.Random(seed)
    return [_collapse((n,) * 3, (1.0 / n,) * 3, (-(n // 2) / n,) * 3, _shape(rng, True)) for n in _scan_grids(case)]


def _fmr_levels(case):
    n = case["nx"]
    return inputs.nested_boxes(n, 1.0 / n, (-(n // 2) / n,) * 3, case["levels"], [case["n_child"]] * (case["levels"] - 1))


def _fmr_states(case, seed):
    shape = _shape(random.Random(seed))
    return [_collapse(lv["n"], lv["h"], lv["x0"], shape) for lv in _fmr_levels(case)]


# ---------------------------------------------------------------------------
# The calls
# ---------------------------------------------------------------------------
def _padded(u, pitch):
    out = torch.zeros((*u.shape[:3], pitch), dtype=torch.float64, device=DEV)
    out[..., : u.shape[3]] = u
    return out.reshape(-1)


def _buffer(nbytes):
    return torch.empty((nbytes + 7) // 8, dtype=torch.float64, device=DEV)


def prepare(case, seed):
    p = C.make_params(**_plain_params(case))
    s = {"case": case, "p": p}
    if case["call"] == "scan":
        s["first"] = [u.reshape(-1) for u in _scan_states(case, seed)]
        ns = _scan_grids(case)
        s["scan"] = BatchScan([C.make_grid(n, 1.0 / n, x0=(-(n // 2) / n,) * 3) for n in ns], p, [CFL / n for n in ns],
                              max_steps=case["steps"], device=DEV, tune=(1, 32, 4, 3))
        s["stream"] = torch.cuda.Stream()  # a scan runs as one captured graph, on a stream of its own
        return s
    if case["call"] == "fmr":
        s["hier"] = Hierarchy(_fmr_levels(case), p, device=DEV)
        s["first"] = [u.reshape(-1) for u in _fmr_states(case, seed)]
        return s
    u = _initial(case, seed)
    s["first"] = _padded(u, case["pitch"])
    h = _spacing(case)
    s["dt"] = CFL * min(h)
    s["grid"] = g = C.make_grid(_n(case), h, x0=tuple(-(v // 2) * d for v, d in zip(_n(case), h)), pitch=case["pitch"])
    if case["call"] in ("adjoint", "vjp"):
        s["lam"] = _padded(_cotangent(case, seed), case["pitch"])
        s["out"] = torch.zeros_like(s["lam"])
        s["ws"] = _buffer(C.cosmos_adjoint_workspace_bytes(
            g, p, C.COSMOS_OP_ADJOINT if case["call"] == "adjoint" else C.COSMOS_OP_VJP))
        if case["call"] == "adjoint":  # the stage states that a forward replay keeps
            s["stages"] = [_padded(y, case["pitch"]) for y in _stages(u, 0.0, s["dt"], h, _plain_params(case))]
        return s
    if case["call"] == "constraints":
        s["hm"] = torch.zeros(4 * C.cosmos_field_stride(g), dtype=torch.float64, device=DEV)
        s["ws"] = _buffer(C.cosmos_workspace_bytes(g, p, C.COSMOS_OP_CONSTRAINTS))
        return s
    s["ev"] = Evolution(g, p, device=DEV)
    s["ev"].state.copy_(s["first"])
    s["out"] = torch.zeros_like(s["first"])
    return s


def _inner(s, flat):
    c = s["case"]
    return flat.view(-1, c["nz"], c["ny"], c["pitch"])[..., : c["nx"]]


def run(s):
    call, p = s["case"]["call"], s["p"]
    steps = s["case"]["steps"]
    if call == "rhs":
        return _inner(s, s["ev"].rhs(0.0, s["out"]))
    if call == "step":  # from the given initial data each time, as a run starts
        s["ev"].state.copy_(s["first"])
        s["ev"].step(0.0, s["dt"], steps)
        return _inner(s, s["ev"].state)
    if call == "scan":
        for u, first in zip(s["scan"].states, s["first"]):
            u.copy_(first)
        s["scan"].run(0, steps, stream=s["stream"])
        torch.cuda.current_stream().wait_stream(s["stream"])
        return s["scan"].states
    if call == "fmr":
        for u, first in zip(s["hier"].states, s["first"]):
            u.copy_(first)
        s["hier"].step(0.0, CFL / s["case"]["nx"], steps)
        return s["hier"].states
    if call == "adjoint":
        C.check(C.cosmos_adjoint_step_stages(s["grid"], p, s["first"], *s["stages"], s["lam"], s["out"], 0.0, s["dt"],
                                             s["ws"]))
        return _inner(s, s["out"])
    if call == "vjp":
        C.check(C.cosmos_rhs_vjp(s["grid"], p, s["first"], s["lam"], s["out"], 0.0, s["ws"]))
        return _inner(s, s["out"])
    norms = (C.ctypes.c_double * 8)()
    C.check(C.cosmos_constraints(s["grid"], p, s["first"], s["hm"], norms, s["ws"]))
    return {"fields": _inner(s, s["hm"]), "norms": torch.tensor(list(norms), dtype=torch.float64)}


def work(case):
    """Bytes: each input state read once and each output written once.  Operations: those of the finite differences
    and of the pointwise algebra of one right-hand side, per point, times the right-hand sides of the call."""
    fluid, scalar = MATTER[case["matter"]]
    nf = 24 + 4 * fluid + 2 * scalar
    rhs = 3300 + 1100 * fluid + 300 * scalar
    if case["call"] == "scan":
        pts, rhss = sum(n ** 3 for n in _scan_grids(case)), 4 * case["steps"]
    elif case["call"] == "fmr":
        size = [lv["n"][0] * lv["n"][1] * lv["n"][2] for lv in _fmr_levels(case)]
        return {"bytes": 16 * nf * sum(size), "flops": 4 * rhs * sum(v * 2 ** l for l, v in enumerate(size))}
    else:
        pts = case["nx"] * case["ny"] * case["nz"]
        rhss = {"rhs": 1, "step": 4 * case["steps"], "adjoint": 4 * 2.6, "vjp": 2.6, "constraints": 0.5}[case["call"]]
    moved = {"adjoint": 6 * nf, "vjp": 3 * nf, "constraints": nf + 4}.get(case["call"], 2 * nf)
    return {"bytes": int(8 * moved * pts), "flops": int(rhs * rhss * pts)}


# ---------------------------------------------------------------------------
# The same in plain torch, FP64 (arrays [field, z, y, x]; axis d is dimension -1 - d)
# ---------------------------------------------------------------------------
def _sh(f, d, o):
    return torch.roll(f, -o, -1 - d)


def _d1(f, d, h):
    return (8.0 * (_sh(f, d, 1) - _sh(f, d, -1)) - (_sh(f, d, 2) - _sh(f, d, -2))) / (12.0 * h[d])


def _d2(f, a, b, h):
    if a != b:
        return _d1(_d1(f, a, h), b, h)
    near = (_sh(f, a, 1) - f) + (_sh(f, a, -1) - f)
    far = (_sh(f, a, 2) - f) + (_sh(f, a, -2) - f)
    return (16.0 * near - far) / (12.0 * h[a] * h[a])


def _dissipation(f, h, sigma):
    out = 0.0
    for d in range(3):
        s = [_sh(f, d, k) + _sh(f, d, -k) for k in (1, 2, 3)]
        out = out + (sigma / (64.0 * h[d])) * ((s[2] - s[1]) - 5.0 * (s[1] - s[0]) + 10.0 * (s[0] - 2.0 * f))
    return out


def _mat(u, first):
    return [[u[first + SYM[i][j]] for j in range(3)] for i in range(3)]


def _inverse(g):
    c = [[g[(i + 1) % 3][(j + 1) % 3] * g[(i + 2) % 3][(j + 2) % 3] - g[(i + 1) % 3][(j + 2) % 3] * g[(i + 2) % 3][(j + 1) % 3]
          for i in range(3)] for j in range(3)]
    det = g[0][0] * c[0][0] + g[0][1] * c[1][0] + g[0][2] * c[2][0]
    return [[c[i][j] / det for j in range(3)] for i in range(3)]


def _geometry(u, h):
    """Conformal metric, its inverse, Christoffels of both kinds, and the Ricci tensor of the physical metric."""
    chi, gt = u[0], _mat(u, 1)
    gu = _inverse(gt)
    dg = [[[None] * 3 for _ in range(3)] for _ in range(3)]  # dg[k][i][j] = d_k gt_ij
    for i, j in PAIRS:
        for k in range(3):
            dg[k][i][j] = dg[k][j][i] = _d1(gt[i][j], k, h)
    low = [[[0.5 * (dg[i][k][j] + dg[j][k][i] - dg[k][i][j]) for j in range(3)] for i in range(3)] for k in range(3)]
    up = [[[sum(gu[k][l] * low[l][i][j] for l in range(3)) for j in range(3)] for i in range(3)] for k in range(3)]
    gd = [sum(gu[i][j] * up[k][i][j] for i in range(3) for j in range(3)) for k in range(3)]
    dG = [[_d1(u[14 + k], i, h) for k in range(3)] for i in range(3)]  # dG[i][k] = d_i Gt^k
    c = [[[sum(gu[m][l] * up[k][l][i] for l in range(3)) for i in range(3)] for m in range(3)] for k in range(3)]
    dchi = [_d1(chi, k, h) for k in range(3)]
    ddchi = [[None] * 3 for _ in range(3)]
    for i, j in PAIRS:
        ddchi[i][j] = ddchi[j][i] = _d2(chi, i, j, h) - sum(up[k][i][j] * dchi[k] for k in range(3))
    lap = sum(gu[i][j] * ddchi[i][j] for i in range(3) for j in range(3))
    sq = sum(gu[i][j] * dchi[i] * dchi[j] for i in range(3) for j in range(3))
    ric = [[None] * 3 for _ in range(3)]
    for i, j in PAIRS:
        r = 0.0
        for l in range(3):
            for m in range(l, 3):
                r = r - (0.5 if l == m else 1.0) * gu[l][m] * _d2(gt[i][j], l, m, h)
        for k in range(3):
            r = r + 0.5 * (gt[k][i] * dG[j][k] + gt[k][j] * dG[i][k]) + 0.5 * gd[k] * (low[i][j][k] + low[j][i][k])
            for m in range(3):
                r = r + c[k][m][i] * low[j][k][m] + c[k][m][j] * low[i][k][m] + c[k][m][i] * low[k][m][j]
        r = r + (ddchi[i][j] + gt[i][j] * lap) / (2.0 * chi) - dchi[i] * dchi[j] / (4.0 * chi * chi) - 3.0 * gt[i][j] * sq / (4.0 * chi * chi)
        ric[i][j] = ric[j][i] = r
    return gt, gu, dg, up, gd, dG, dchi, ric


def _raise(gu, v):
    return [sum(gu[i][j] * v[j] for j in range(3)) for i in range(3)]


def _dot(a, b):
    return sum(x * y for x, y in zip(a, b))


def _primitives(u, w):
    """rho, v_i of the fluid from the conserved fields."""
    chi, gu = u[0], _inverse(_mat(u, 1))
    c32 = chi * torch.sqrt(chi)
    E, J = u[24] * c32, [u[25 + i] * c32 for i in range(3)]
    D = E * E - chi * _dot(_raise(gu, J), J)
    a = (1.0 - w) * E
    rho = 2.0 * D / (a + torch.sqrt(a * a + 4.0 * w * D))
    return rho, [j / (E + w * rho) for j in J]


def _minmod(a, b):
    z = torch.zeros_like(a)
    both = torch.where((a > 0) & (b > 0), torch.where(a <= b, a, b), z)
    return torch.where((a < 0) & (b < 0), torch.where(a >= b, a, b), both)


def _face_flux(u, prim, d, w):
    """Kurganov-Tadmor flux through the face between each cell and its neighbour along axis d."""
    mean = lambda f: 0.5 * (f + _sh(f, d, 1))  # noqa: E731
    chi, alpha, beta = mean(u[0]), mean(u[17]), mean(u[18 + d])
    gu = [[chi * v for v in row] for row in _inverse(_mat([mean(u[f]) for f in range(7)], 1))]
    left, right = [], []
    for q in [prim[0]] + prim[1]:
        step = _sh(q, d, 1) - q
        slope = _minmod(_sh(step, d, -1), step)
        left.append(q + 0.5 * slope)
        right.append(_sh(q - 0.5 * slope, d, 1))
    U, F, speed = [], [], []
    for rho, *v in (left, right):
        vu = _raise(gu, v)
        v2 = _dot(vu, v)
        hw, P = (1.0 + w) * rho / (1.0 - v2), w * rho
        U.append([hw - P] + [hw * x for x in v])
        F.append([alpha * hw * vu[d] - beta * (hw - P)] +
                 [alpha * (hw * vu[d] * v[i] + (P if i == d else 0.0)) - beta * hw * v[i] for i in range(3)])
        root = torch.sqrt(w * (1.0 - v2) * (gu[d][d] * (1.0 - v2 * w) - vu[d] * vu[d] * (1.0 - w)))
        for sign in (1.0, -1.0):
            speed.append(torch.abs(alpha / (1.0 - v2 * w) * (vu[d] * (1.0 - w) + sign * root) - beta))
    a = speed[0]
    for x in speed[1:]:
        a = torch.where(a >= x, a, x)
    half = 0.5 / (chi * torch.sqrt(chi))
    return [half * (F[0][m] + F[1][m] - a * (U[1][m] - U[0][m])) for m in range(4)]


def _sources(u, gu, gt, h, p, prim):
    """rho_H, J_i, S_ij (lists) of fluid and scalar together."""
    chi = u[0]
    E, J, S = 0.0, [0.0] * 3, [[0.0] * 3 for _ in range(3)]
    fl = sc = None
    if p["fluid"]:
        c32 = chi * torch.sqrt(chi)
        E, J, P = u[24] * c32, [u[25 + i] * c32 for i in range(3)], p["w"] * prim[0]
        S = [[J[i] * J[j] / (E + P) + P * gt[i][j] / chi for j in range(3)] for i in range(3)]
        fl = (E, J, [row[:] for row in S])
    if p["scalar"]:
        f = 24 + 4 * p["fluid"]
        Pi, dphi = u[f + 1], [_d1(u[f], k, h) for k in range(3)]
        grad = chi * _dot(_raise(gu, dphi), dphi)
        E, J = E + 0.5 * (Pi * Pi + grad), [J[i] + Pi * dphi[i] for i in range(3)]
        S = [[S[i][j] + dphi[i] * dphi[j] - 0.5 * (grad - Pi * Pi) * gt[i][j] / chi for j in range(3)] for i in range(3)]
        sc = (f, Pi, dphi)
    return E, J, S, fl, sc


def _rhs(u, t, h, p):
    """The right-hand side of all fields of `u` (a tensor [field, z, y, x])."""
    gt, gu, dg, up, gd, dG, dchi, ric = _geometry(u, h)
    chi, K, At, alpha = u[0], u[7], _mat(u, 8), u[17]
    beta, B = [u[18 + i] for i in range(3)], [u[21 + i] for i in range(3)]
    Kref = -3.0 * p["H0"] / (1.0 + 1.5 * (1.0 + p["w"]) * p["H0"] * (t - p["t0"]))
    prim = _primitives(u, p["w"]) if p["fluid"] else None
    matter = p["fluid"] or p["scalar"]
    E, J, S, fl, sc = _sources(u, gu, gt, h, p, prim)
    da = [_d1(alpha, k, h) for k in range(3)]
    db = [[_d1(beta[i], k, h) for i in range(3)] for k in range(3)]  # db[k][i] = d_k beta^i
    div = db[0][0] + db[1][1] + db[2][2]
    adv = lambda f: sum(beta[k] * _d1(f, k, h) for k in range(3))  # noqa: E731
    out = [None] * u.shape[0]
    out[0] = adv(chi) + (2.0 / 3.0) * chi * (alpha * K - div)
    Aup = [[sum(gu[i][k] * At[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
    A2 = [[sum(Aup[i][k] * gu[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
    AA = sum(A2[i][j] * At[i][j] for i in range(3) for j in range(3))
    dd = [[None] * 3 for _ in range(3)]
    X = [[None] * 3 for _ in range(3)]
    mixed = _dot(_raise(gu, dchi), da)
    for i, j in PAIRS:
        dd[i][j] = dd[j][i] = _d2(alpha, i, j, h) - sum(up[k][i][j] * da[k] for k in range(3))
        hess = dd[i][j] + (dchi[i] * da[j] + dchi[j] * da[i] - gt[i][j] * mixed) / (2.0 * chi)
        X[i][j] = X[j][i] = alpha * (ric[i][j] - 8.0 * math.pi * S[i][j]) - hess
    lap = chi * sum(gu[i][j] * dd[i][j] for i in range(3) for j in range(3)) - 0.5 * mixed
    out[7] = adv(K) - lap + alpha * (AA + K * K / 3.0)
    if matter:
        trS = chi * sum(gu[i][j] * S[i][j] for i in range(3) for j in range(3))
        out[7] = out[7] + 4.0 * math.pi * alpha * (E + trS)
    trX = sum(gu[i][j] * X[i][j] for i in range(3) for j in range(3))
    for m, (i, j) in enumerate(PAIRS):
        out[1 + m] = (adv(gt[i][j]) - 2.0 * alpha * At[i][j] - (2.0 / 3.0) * gt[i][j] * div +
                      sum(gt[i][k] * db[j][k] + gt[j][k] * db[i][k] for k in range(3)))
        out[8 + m] = (adv(At[i][j]) - (2.0 / 3.0) * At[i][j] * div + chi * (X[i][j] - gt[i][j] * trX / 3.0) +
                      alpha * (K * At[i][j] - 2.0 * sum(At[i][k] * Aup[k][j] for k in range(3))) +
                      sum(At[i][k] * db[j][k] + At[j][k] * db[i][k] for k in range(3)))
    del X, dd, ric
    ddiv = [sum(_d2(beta[k], j, k, h) for k in range(3)) for j in range(3)]
    dK = [_d1(K, k, h) for k in range(3)]
    for i in range(3):
        s = sum((1.0 if a == b else 2.0) * gu[a][b] * _d2(beta[i], a, b, h) for a, b in PAIRS) + _dot(gu[i], ddiv) / 3.0
        s = s - sum(gd[k] * db[k][i] for k in range(3)) + (2.0 / 3.0) * gd[i] * div - 2.0 * _dot(A2[i], da)
        s = s + 2.0 * alpha * (sum(up[i][j][k] * A2[j][k] for j in range(3) for k in range(3)) -
                               1.5 * _dot(A2[i], dchi) / chi - (2.0 / 3.0) * _dot(gu[i], dK))
        if matter:
            s = s - 16.0 * math.pi * alpha * _dot(gu[i], J)
        out[14 + i] = adv(u[14 + i]) + s
        out[18 + i] = adv(beta[i]) + 0.75 * B[i] if p["shift"] else torch.zeros_like(chi)
        out[21 + i] = adv(B[i]) + s - p["eta"] * B[i] if p["shift"] else torch.zeros_like(chi)
    out[17] = adv(alpha) - (2.0 * alpha if p["slicing"] == 0 else alpha * alpha) * (K - Kref)
    if p["fluid"]:
        E, J, Sf = fl
        root = 1.0 / (chi * torch.sqrt(chi))
        Sm = [[sum(gu[i][k] * Sf[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
        Su = [[chi * chi * sum(Sm[i][k] * gu[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
        SK = sum(Su[i][j] * (At[i][j] + gt[i][j] * K / 3.0) for i in range(3) for j in range(3)) / chi
        out[24] = root * (alpha * SK - chi * _dot(_raise(gu, J), da))
        for i in range(3):
            dgam = sum(Su[a][b] * (dg[i][a][b] / chi - gt[a][b] * dchi[i] / (chi * chi)) for a in range(3) for b in range(3))
            out[25 + i] = root * (_dot(J, db[i]) - E * da[i] + 0.5 * alpha * dgam)
        for d in range(3):
            for m, F in enumerate(_face_flux(u, prim, d, p["w"])):
                out[24 + m] = out[24 + m] - (F - _sh(F, d, -1)) / h[d]
    if p["scalar"]:
        f, Pi, dphi = sc
        ddphi = sum((1.0 if a == b else 2.0) * gu[a][b] * _d2(u[f], a, b, h) for a, b in PAIRS)
        lap = chi * (ddphi - _dot(gd, dphi)) - 0.5 * _dot(_raise(gu, dchi), dphi)
        out[f] = adv(u[f]) - alpha * Pi
        out[f + 1] = adv(Pi) + alpha * (K * Pi - lap) - chi * _dot(_raise(gu, dphi), da)
    return torch.stack([out[f] if p["fluid"] and 24 <= f < 28 else out[f] + _dissipation(u[f], h, p["ko_sigma"])
                        for f in range(u.shape[0])])


def _stages(u, t, dt, h, p, full=False, fix=None):
    """The stage states U_2, U_3, U_4 of one RK4 step (and the new state with `full`); fix(stage, state) sets the
    ghost points of each stage state of a refined level."""
    fix = fix or (lambda stage, y: y)
    u = fix(1, u)
    k = _rhs(u, t, h, p)
    acc, y2 = k, fix(2, u + 0.5 * dt * k)
    k = _rhs(y2, t + 0.5 * dt, h, p)
    acc, y3 = acc + 2.0 * k, fix(3, u + 0.5 * dt * k)
    k = _rhs(y3, t + 0.5 * dt, h, p)
    acc, y4 = acc + 2.0 * k, fix(4, u + dt * k)
    if not full:
        return y2, y3, y4
    return u, y2, y3, y4, u + (dt / 6.0) * (acc + _rhs(y4, t + dt, h, p))


def _pull_back(u, w, t, h, p):
    """(d rhs / d u)^T w."""
    x = u.detach().clone().requires_grad_(True)
    return torch.autograd.grad(_rhs(x, t, h, p), x, w)[0]


def _constraints(u, h, p):
    gt, gu, dg, up, gd, dG, dchi, ric = _geometry(u, h)
    chi, K, At = u[0], u[7], _mat(u, 8)
    prim = _primitives(u, p["w"]) if p["fluid"] else None
    E, J, _, _, _ = _sources(u, gu, gt, h, p, prim)
    Aup = [[sum(gu[i][k] * At[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
    A2 = [[sum(Aup[i][k] * gu[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
    R = chi * sum(gu[i][j] * ric[i][j] for i in range(3) for j in range(3))
    v = [R + (2.0 / 3.0) * K * K - sum(A2[i][j] * At[i][j] for i in range(3) for j in range(3)) - 16.0 * math.pi * E]
    low = []
    for k in range(3):
        s = 0.0
        for j in range(3):
            for l in range(3):
                s = s + gu[j][l] * (_d1(At[k][l], j, h) - sum(up[m][j][k] * At[m][l] + up[m][j][l] * At[k][m] for m in range(3)))
        low.append(s - (2.0 / 3.0) * _d1(K, k, h) - 8.0 * math.pi * J[k])
    v += [_dot(gu[i], low) - 1.5 * _dot(A2[i], dchi) / chi for i in range(3)]
    v = torch.stack(v)
    return v, torch.cat([torch.sqrt((v * v).mean(dim=(1, 2, 3))), v.abs().amax(dim=(1, 2, 3))])


# ---- a refined hierarchy: ghost values from the parent's step, two half steps per parent step, injection ----
_W6 = (3.0 / 256.0, -25.0 / 256.0, 150.0 / 256.0, 150.0 / 256.0, -25.0 / 256.0, 3.0 / 256.0)


def _interpolate(parent, lv):
    """The parent's field values at the points of a child level, one axis at a time."""
    out = parent
    for d in range(3):
        pos = [lv["origin"][d] + i for i in range(lv["n"][d])]
        n = out.shape[-1 - d]
        even = torch.tensor([x % 2 == 0 for x in pos], device=DEV)
        taps = [out.index_select(-1 - d, torch.tensor([(x // 2 + o) % n for x in pos], device=DEV)) for o in range(-2, 4)]
        half = sum(w * v for w, v in zip(_W6, taps))
        out = torch.where(even.view([-1 if q == 3 - d else 1 for q in range(4)]), taps[2], half)
    return out


def _inside(lv):
    return (slice(None),) + tuple(slice(lv["lo"][d], lv["hi"][d]) for d in (2, 1, 0))


def _with_ghosts(u, parent, lv):
    out = _interpolate(parent, lv)
    out[_inside(lv)] = u[_inside(lv)]
    return out


def _stage_value(step, theta, stage):
    """The parent's solution at a child's stage: RK4's continuous extension and its derivatives, r = 1/2."""
    un, y2, y3, y4, u1 = step
    q, r = theta, 0.5
    b = [q - 1.5 * q ** 2 + 2 / 3 * q ** 3, q ** 2 - 2 / 3 * q ** 3, q ** 2 - 2 / 3 * q ** 3, -0.5 * q ** 2 + 2 / 3 * q ** 3]
    d1 = [1 - 3 * q + 2 * q ** 2, 2 * q - 2 * q ** 2, 2 * q - 2 * q ** 2, -q + 2 * q ** 2]
    d2, d3 = [4 * q - 3, 2 - 4 * q, 2 - 4 * q, 4 * q - 1], [4.0, -4.0, -4.0, 4.0]
    e1, e2, e3 = [(0, 0, 0), (0.5, 0, 0), (0.5, 0.25, 0), (1, 0.5, 0.25)][stage - 1]
    k = [x + e1 * r * y + e2 * r ** 2 * z + e3 * r ** 3 * v for x, y, z, v in zip(b, d1, d2, d3)]
    # dt k_1 = 2 (y2 - un), dt k_2 = 2 (y3 - un), dt k_3 = y4 - un, dt k_4 = 6 (u1 - un) - dt (k_1 + 2 k_2 + 2 k_3)
    return (un + (2 * k[0] - 2 * k[3]) * (y2 - un) + (2 * k[1] - 4 * k[3]) * (y3 - un) + (k[2] - 2 * k[3]) * (y4 - un) +
            6 * k[3] * (u1 - un))


def _advance(U, levels, l, t, dt, theta, parent_step, p):
    lv = levels[l]
    fix = (lambda s, y: _with_ghosts(y, _stage_value(parent_step, theta, s), lv)) if l else None
    step = _stages(U[l], t, dt, lv["h"], p, full=True, fix=fix)
    if l:  # the fluid's ghost points may hold anything from here on: they are set before they are read
        step = step[:4] + (_with_ghosts(step[4], parent_step[4], lv),)
    U[l] = step[4]
    if l + 1 < len(levels):
        child = levels[l + 1]
        for half in range(2):
            _advance(U, levels, l + 1, t + 0.5 * half * dt, 0.5 * dt, 0.5 * half, step, p)
        first = [child["lo"][d] + (child["origin"][d] + child["lo"][d]) % 2 for d in range(3)]
        pick = tuple(slice(first[d], child["hi"][d], 2) for d in (2, 1, 0))
        at = [torch.tensor([(child["origin"][d] + i) // 2 % lv["n"][d] for i in range(first[d], child["hi"][d], 2)], device=DEV)
              for d in (2, 1, 0)]
        U[l] = U[l].clone()
        U[l][:, at[0][:, None, None], at[1][None, :, None], at[2][None, None, :]] = U[l + 1][(slice(None),) + pick]


@torch.no_grad()
def exact(case, seed):
    p, call = _plain_params(case), case["call"]
    if call == "scan":
        out = []
        for n, u in zip(_scan_grids(case), _scan_states(case, seed)):
            for s in range(case["steps"]):
                u = _stages(u, s * CFL / n, CFL / n, (1.0 / n,) * 3, p, full=True)[4]
            out.append(u.reshape(-1))
        return out
    if call == "fmr":
        levels, U = _fmr_levels(case), _fmr_states(case, seed)
        for s in range(case["steps"]):
            _advance(U, levels, 0, s * CFL / case["nx"], CFL / case["nx"], 0.0, None, p)
            for l in range(1, len(levels)):
                U[l] = _with_ghosts(U[l], U[l - 1], levels[l])
        return [u.reshape(-1) for u in U]
    u, h = _initial(case, seed), _spacing(case)
    dt = CFL * min(h)
    if call == "rhs":
        return _rhs(u, 0.0, h, p)
    if call == "step":
        for s in range(case["steps"]):
            u = _stages(u, s * dt, dt, h, p, full=True)[4]
        return u
    if call == "constraints":
        fields, norms = _constraints(u, h, p)
        return {"fields": fields, "norms": norms.cpu()}
    with torch.enable_grad():
        w = _cotangent(case, seed)
        if call == "vjp":
            return _pull_back(u, w, 0.0, h, p)
        with torch.no_grad():
            y = _stages(u, 0.0, dt, h, p)
        v4 = _pull_back(y[2], (dt / 6.0) * w, dt, h, p)
        v3 = _pull_back(y[1], (dt / 3.0) * w + dt * v4, 0.5 * dt, h, p)
        v2 = _pull_back(y[0], (dt / 3.0) * w + 0.5 * dt * v3, 0.5 * dt, h, p)
        v1 = _pull_back(u, (dt / 6.0) * w + 0.5 * dt * v2, 0.0, h, p)
        return w + v1 + v2 + v3 + v4
