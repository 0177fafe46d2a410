"""Pointwise BSSN + matter algebra, stated in the expression DSL.

This is the GPU path's own statement of the evolution equations of the paper
(section "Physical system settings": Einstein equations with T = T^SC + T^FL,
P = w rho, box phi = 0, div T^FL = 0), rewritten in the standard BSSN
(chi-variant) form that the paper defers to numerical-relativity textbooks.
It is turned into straight-line CUDA by ``generate.py``.

Inputs at one grid point (layout shared with the stencil kernels):
  in[0 .. NF)                        field values (state order)
  in[NF + 3 m + k]                   d_k of the m-th first-derivative field
  in[NF + 3 ND1 + 6 m + p]           second derivative p = xx,xy,xz,yy,yz,zz
                                     of the m-th second-derivative field
  in[NF + 3 ND1 + 6 ND2]             fluid rest-frame density rho (fluid only)
First-derivative fields: the 24 BSSN fields, then phi, Pi (scalar on).
Second-derivative fields: chi, gt_xx..gt_zz, alpha, beta^x..z, then phi.

Outputs: out[f] = d_t of field f WITHOUT the Kreiss-Oliger term and, for the
fluid fields, without the flux divergence (geometric sources only).

Runtime parameters (struct AlgebraParams): eta (Gamma-driver damping),
Kref (background trace K_ref(t) of the stage time), lapse_c1, lapse_c2
(d_t alpha = beta.d alpha - alpha (c1 + c2 alpha)(K - Kref): 1+log is
c1=2, c2=0; harmonic is c1=0, c2=1), shift_on (1 Gamma-driver, 0 frozen),
w (equation of state).

The pass that evaluates this is bound by the FP64 pipe, so the expressions are
grouped for few FP64 instructions (a multiply that feeds one add is free):
factors 1/2 and 2 are folded into quantities formed once, the equal terms of
diagonal components are formed once, terms that one tensor multiplies are
summed before it does, and what the trace-free projection removes is not
formed.  Vacuum: 803 multiply-adds per point (753 products, 633 sums)
against 973 for the textbook grouping, fluid 925 against 1148, reverse mode
2071 against 2480, constraints 556 against 777; a 256^3 vacuum RK4 step went
from 169.0 to 153.3 ms and a 128^3 fluid one from 39.1 to 36.3 ms.  The stage
kernel's form (inverse metric, 1/chi and the advection formed elsewhere) has 718
in vacuum, 840 with the fluid.
"""
from __future__ import annotations

import math

from .expr import Graph, sqrt

PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
PIDX = {(0, 0): 0, (0, 1): 1, (0, 2): 2, (1, 0): 1, (1, 1): 3, (1, 2): 4, (2, 0): 2, (2, 1): 4, (2, 2): 5}

CHI, GT, TRK, AT, GAM, ALP, BET, BB = 0, 1, 7, 8, 14, 17, 18, 21
D2_FIELDS_BSSN = [CHI, 1, 2, 3, 4, 5, 6, ALP, BET, BET + 1, BET + 2]


def layout(fluid: bool, scalar: bool):
    nf = 24 + 4 * fluid + 2 * scalar
    d1 = list(range(24))
    d2 = list(D2_FIELDS_BSSN)
    if scalar:
        s = 24 + 4 * fluid
        d1 += [s, s + 1]
        d2 += [s]
    names = [f"u{f}" for f in range(nf)]
    names += [f"d{f}_{k}" for f in d1 for k in range(3)]
    names += [f"dd{f}_{p}" for f in d2 for p in range(6)]
    if fluid:
        names += ["rho"]
    return dict(nf=nf, d1=d1, d2=d2, names=names, nin=len(names))


class Sym:
    """Symmetric 3x3 tensor of expressions stored as 6 components."""

    def __init__(self, c):
        self.c = list(c)

    def __getitem__(self, ij):
        return self.c[PIDX[ij]]


def contract_sym(Mu, N):
    """sum_ij M^ij N_ij for symmetric M, N (M given with doubled off-diagonals)."""
    s = None
    for m, (i, j) in enumerate(PAIRS):
        t = Mu[m] * N[(i, j)]
        s = t if s is None else s + t
    return s


def split_layout(fluid: bool, scalar: bool):
    """Input slots of the split form (``algebra(..., split=True)``): region A holds
    what the first phase reads, region B what the second one does and the slots
    ``r{f}`` that take the outputs of fields without a slot of their own there.

    Per field with second derivatives ten slots (d_k, dd_p, m), per field with
    first derivatives four (d_k, m), a field whose derivatives only advect it has
    m alone: its whole advection with the dissipation term (that of the metric
    and Gamma is read at the end of the first phase).  The inverse metric gu, 1/chi
    (ichi) and kdiff = K - Kref are formed outside; the shift's slots serve the
    advections, the algebra does not read them.  ``out`` =
    the region-B slot that takes output f: its m slot (read by that output alone)
    or r{f}.

    Units: lengths in l (the algebra does not see its value but through the
    parameters below).  u of K, At, Pi carries l, u of the fluid fields and rho
    l^2, m the units of its output; differences, u of B^i and kdiff come without
    the l of their field, which the parameters that multiply them hold: len = l,
    c75 = 3/4 l, c43 = 4/3 l, eta l^2, lapse_c1 l, lapse_c2 l.  out[f] carries one l
    more than field f.

    The raised At is formed in the first phase (both phases then take about as
    long as the differences of the other region), except with the fluid, whose
    own quantities already fill the registers between the phases."""

    def d2(f):
        return [f"d{f}_{k}" for k in range(3)] + [f"dd{f}_{p}" for p in range(6)] + [f"m{f}"]

    def d1(f):
        return [f"d{f}_{k}" for k in range(3)] + [f"m{f}"]

    a, b = [], []
    for f in range(GT, GT + 6):
        a += d2(f)
    for f in range(GAM, GAM + 3):
        a += d1(f)
    early = not fluid
    a += [f"u{f}" for f in [*range(GT, GT + 6), *range(BET, BET + 3)]] + [f"gu{m}" for m in range(6)]
    a += [f"u{f}" for f in range(AT, AT + 6)] * early
    if fluid:
        a += ["u0", "u24", "u25", "u26", "u27", "rho"]
    ph = 24 + 4 * fluid
    for f in [CHI, ALP, BET, BET + 1, BET + 2] + [ph] * scalar:
        b += d2(f)
    b += d1(TRK)
    b += [f"m{f}" for f in [*range(AT, AT + 6), *range(BB, BB + 3)] + [ph + 1] * scalar]
    b += [f"u{f}" for f in [*range(0, GAM), ALP, *range(BB, BB + 3)]] + ["kdiff", "ichi"]
    if fluid:
        b += ["u24", "u25", "u26", "u27", "rho"]
    if scalar:
        b += [f"u{ph + 1}"]
    b += [f"r{f}" for f in [*range(GT, GT + 6), *range(GAM, GAM + 3)] + [24, 25, 26, 27] * fluid]
    nf = 24 + 4 * fluid + 2 * scalar
    out = [b.index(next(x for x in (f"m{f}", f"r{f}") if x in b)) for f in range(nf)]
    return dict(a=a, b=b, out=out, early=early)


def algebra(fluid: bool, scalar: bool, split: bool = False):
    """The right-hand side as a graph: (graph, layout, outputs).

    With ``split`` the outputs contain the dissipation terms, the inputs are
    those of ``split_layout``, and the graph carries ``cut``: the nodes that end
    the first phase, whose inputs are those of region A."""
    g = Graph()
    L = layout(fluid, scalar)
    nf = L["nf"]
    cut = []
    u = [g.input(f"u{f}") for f in range(nf)]

    def d(f, k):
        return g.input(f"d{f}_{k}")

    def dd(f, i, j):
        return g.input(f"dd{f}_{PIDX[(i, j)]}")

    eta = g.param("eta")
    if split:
        ulen, c75, c43 = g.param("len"), g.param("c75"), g.param("c43")
    else:
        Kref = g.param("Kref")
        ulen, c75, c43 = 1.0, 0.75, 4.0 / 3.0
    c1, c2, shift_on, w = g.param("lapse_c1"), g.param("lapse_c2"), g.param("shift_on"), g.param("w")
    pi = math.pi

    chi, K, alpha = u[CHI], u[TRK], u[ALP]
    gt = Sym(u[GT:GT + 6])
    At = Sym(u[AT:AT + 6])
    Gt = u[GAM:GAM + 3]
    beta = u[BET:BET + 3]
    B = u[BB:BB + 3]
    dchi = [d(CHI, k) for k in range(3)]
    dK = [d(TRK, k) for k in range(3)]
    dal = [d(ALP, k) for k in range(3)]

    def dgt(k, i, j):
        return d(GT + PIDX[(i, j)], k)

    def dAt(k, i, j):
        return d(AT + PIDX[(i, j)], k)

    def dGt(k, i):
        return d(GAM + i, k)

    def dbeta(k, i):
        return d(BET + i, k)

    def dB(k, i):
        return d(BB + i, k)

    def ddgt(l, m, i, j):
        return dd(GT + PIDX[(i, j)], l, m)

    # ---- inverse conformal metric (cofactors / det) ----
    c00 = gt[1, 1] * gt[2, 2] - gt[1, 2] * gt[1, 2]
    c01 = gt[0, 2] * gt[1, 2] - gt[0, 1] * gt[2, 2]
    c02 = gt[0, 1] * gt[1, 2] - gt[0, 2] * gt[1, 1]
    c11 = gt[0, 0] * gt[2, 2] - gt[0, 2] * gt[0, 2]
    c12 = gt[0, 1] * gt[0, 2] - gt[0, 0] * gt[1, 2]
    c22 = gt[0, 0] * gt[1, 1] - gt[0, 1] * gt[0, 1]
    idet = (gt[0, 0] * c00 + gt[0, 1] * c01 + gt[0, 2] * c02).rcp()
    gu = Sym([g.input(f"gu{m}") if split else c * idet for m, c in enumerate([c00, c01, c02, c11, c12, c22])])
    gu2 = [gu[i, j] * (1.0 if i == j else 2.0) for (i, j) in PAIRS]  # doubled off-diagonals
    ichi = g.input("ichi") if split else chi.rcp()

    # ---- Christoffels.  Gl2[k][(i,j)] = 2 Gamma_kij (first kind, doubled: the
    # factors 1/2 cost nothing where they are folded into factors formed once) ----
    Gl2 = []
    for k in range(3):
        row = []
        for (i, j) in PAIRS:
            if i == k:
                row.append(dgt(j, k, k))
            elif j == k:
                row.append(dgt(i, k, k))
            elif i == j:
                row.append(2.0 * dgt(i, k, i) - dgt(k, i, i))
            else:
                row.append(dgt(i, k, j) + dgt(j, k, i) - dgt(k, i, j))
        Gl2.append(Sym(row))
    # second kind Gu[k][(i,j)] = gt^kl Gamma_lij
    hgu = Sym([0.5 * x for x in gu.c])
    Gu = []
    for k in range(3):
        Gu.append(Sym([hgu[k, 0] * Gl2[0][i, j] + hgu[k, 1] * Gl2[1][i, j] + hgu[k, 2] * Gl2[2][i, j]
                       for (i, j) in PAIRS]))

    # ---- conformal Ricci tensor, doubled ----
    # R_ij = -1/2 gt^lm d_l d_m gt_ij + gt_k(i d_j) Gt^k + Gd^k Gamma_(ij)k
    #        + (T_ij + T_ji) + U_ij,
    # T_ij = sum_km C[k][m][i] Gamma_jkm, U_ij = sum_km C[k][m][i] Gamma_kmj,
    # C[k][m][i] = gt^ml Gamma^k_li.  T_ij + U_ij = V_ij = sum_km C[k][m][i] d_m gt_jk
    # (Gamma_jkm + Gamma_kjm = d_m gt_jk), so the quadratic part is V_ij + T_ji: 15
    # products instead of 21 off the diagonal.  The Christoffel products are
    # accumulated into the six components index i by index i, so that only the
    # nine C[.][.][i] of one i exist at a time (fewer values live at once).
    accT, accV = [None] * 6, [None] * 6  # 2 T_ji (i <= j), V_ij
    for i in range(3):
        Ci = [[gu[m, 0] * Gu[k][0, i] + gu[m, 1] * Gu[k][1, i] + gu[m, 2] * Gu[k][2, i] for m in range(3)]
              for k in range(3)]
        # Gamma_jkm is symmetric in k, m: T_ij sums (C[k][m][i] + C[m][k][i]) Gamma_jkm over k <= m
        Cs = {(k, m): (Ci[k][m] if k == m else Ci[k][m] + Ci[m][k]) for (k, m) in PAIRS}
        for j in range(3):
            if j <= i:  # T_ij into R_ji
                s = None
                for (k, m) in PAIRS:
                    t = Cs[(k, m)] * Gl2[j][k, m]
                    s = t if s is None else s + t
                accT[PIDX[(i, j)]] = s
            if j >= i:
                s = None
                for k in range(3):
                    for m in range(3):
                        t = Ci[k][m] * dgt(m, j, k)
                        s = t if s is None else s + t
                accV[PIDX[(i, j)]] = s
    acc = [accT[m] + 2.0 * accV[m] for m in range(6)]
    Gd = [contract_sym(gu2, Gu[k]) for k in range(3)]
    # 2 R_ij as one flat sum:
    #   -gt^lm d_l d_m gt_ij + gt_ki d_j Gt^k + gt_kj d_i Gt^k + Gd^k d_k gt_ij + acc
    # (Gamma_ijk + Gamma_jik = d_k gt_ij); on the diagonal the two equal terms are formed once
    lgt = Sym([ulen * x for x in gt.c])
    Ric2 = []
    for m, (i, j) in enumerate(PAIRS):
        r = acc[m]
        for q, (l, n) in enumerate(PAIRS):
            r = r - gu2[q] * ddgt(l, n, i, j)
        if i == j:
            r = r + 2.0 * (lgt[0, i] * dGt(i, 0) + lgt[1, i] * dGt(i, 1) + lgt[2, i] * dGt(i, 2))
        else:
            for k in range(3):
                r = r + lgt[k, i] * dGt(j, k) + lgt[k, j] * dGt(i, k)
        for k in range(3):
            r = r + Gd[k] * dgt(k, i, j)
        Ric2.append(r)

    # ---- lapse and conformal-factor terms of the trace-free part ----
    # R_ij of the chi part and D_i D_j alpha enter the equation of At_ij through
    # the trace-free part of X_ij = alpha R_ij - D_i D_j alpha - 8 pi alpha S_ij
    # only, so every term proportional to gt_ij is left out of X.  With
    # h = 1/(2 chi):
    #   X_ij = (alpha/2) 2R~_ij + alpha h d_i d_j chi - d_i d_j alpha
    #          + Gamma^k_ij (d_k alpha - alpha h d_k chi)
    #          - h d_i chi w_j - h d_j chi w_i,   w_i = d_i alpha + (alpha h/2) d_i chi
    half_ichi = 0.5 * ichi
    half_alpha = 0.5 * alpha
    ah = alpha * half_ichi
    v = [dal[k] - ah * dchi[k] for k in range(3)]
    Gu_v = [Gu[0][i, j] * v[0] + Gu[1][i, j] * v[1] + Gu[2][i, j] * v[2] for (i, j) in PAIRS]
    hah = 0.5 * ah
    wal = [dal[k] + hah * dchi[k] for k in range(3)]
    hchi = [half_ichi * dchi[k] for k in range(3)]

    # ---- raised At ----
    Aud = [[gu[i, 0] * At[0, j] + gu[i, 1] * At[1, j] + gu[i, 2] * At[2, j] for j in range(3)] for i in range(3)]
    Atu = Sym([Aud[i][0] * gu[0, j] + Aud[i][1] * gu[1, j] + Aud[i][2] * gu[2, j] for (i, j) in PAIRS])
    Atu2 = [Atu[a, b] * (1.0 if a == b else 2.0) for (a, b) in PAIRS]
    GA = [contract_sym(Atu2, Gu[i]) for i in range(3)]
    AA = contract_sym(Atu2, At)

    # ---- Laplacian of the lapse ----
    wchi = [gu[l, 0] * dchi[0] + gu[l, 1] * dchi[1] + gu[l, 2] * dchi[2] for l in range(3)]  # gt^lm d_m chi
    dchi_dal = wchi[0] * dal[0] + wchi[1] * dal[1] + wchi[2] * dal[2]
    lap_a = chi * (contract_sym(gu2, Sym([dd(ALP, i, j) for (i, j) in PAIRS]))
                   - (Gd[0] * dal[0] + Gd[1] * dal[1] + Gd[2] * dal[2])) - 0.5 * dchi_dal

    # ---- matter: rho_H, J_i, the trace S, and Sl_ij = S_ij less its part along gt_ij ----
    rhoH = None
    Jl = [None, None, None]
    Sl = [None] * 6
    Str = None
    fl = {}
    if fluid:
        q = 24
        tau, St = u[q], u[q + 1:q + 4]
        sq = sqrt(chi)
        chi32 = chi * sq  # 1/sqrt(gamma)
        isg = chi32.rcp()  # sqrt(gamma)
        E = tau * chi32
        J = [St[i] * chi32 for i in range(3)]
        wJ = [gu[i, 0] * J[0] + gu[i, 1] * J[1] + gu[i, 2] * J[2] for i in range(3)]  # gt^ij J_j
        J2 = chi * (wJ[0] * J[0] + wJ[1] * J[1] + wJ[2] * J[2])
        rho = g.input("rho")
        P = w * rho
        iEP = (E + P).rcp()
        # S_ij = J_i J_j/(E + P) + P gt_ij/chi
        Jq = [J[i] * iEP for i in range(3)]
        Sl = [Jq[i] * J[j] for (i, j) in PAIRS]
        rhoH = E
        Jl = list(J)
        Sf_tr = J2 * iEP + 3.0 * P
        Str = Sf_tr
        fl = dict(E=E, J=J, wJ=wJ, isg=isg, P=P, iEP=iEP, Str=Sf_tr)
    if scalar:
        s = 24 + 4 * fluid
        Pi_ = u[s + 1]
        dphi = [d(s, k) for k in range(3)]
        wphi = [gu[i, 0] * dphi[0] + gu[i, 1] * dphi[1] + gu[i, 2] * dphi[2] for i in range(3)]
        dphi2 = chi * (wphi[0] * dphi[0] + wphi[1] * dphi[1] + wphi[2] * dphi[2])
        Pi2 = Pi_ * Pi_
        r_sc = 0.5 * (Pi2 + dphi2)
        rhoH = r_sc if rhoH is None else rhoH + r_sc
        for i in range(3):
            Jl[i] = Pi_ * dphi[i] if Jl[i] is None else Jl[i] + Pi_ * dphi[i]
        for m, (i, j) in enumerate(PAIRS):
            t = dphi[i] * dphi[j]
            Sl[m] = t if Sl[m] is None else Sl[m] + t
        t = 1.5 * Pi2 - 0.5 * dphi2
        Str = t if Str is None else Str + t
    have_matter = fluid or scalar

    # ---- right-hand sides ----
    out = [None] * nf
    divb = dbeta(0, 0) + dbeta(1, 1) + dbeta(2, 2)

    def adv(f):
        """Advection of field f; in the split form with its dissipation term, in the units of the output."""
        if split:
            return g.input(f"m{f}")
        return beta[0] * d(f, 0) + beta[1] * d(f, 1) + beta[2] * d(f, 2)

    third_div = (1.0 / 3.0) * divb
    out[CHI] = adv(CHI) + (2.0 * chi) * ((1.0 / 3.0) * (alpha * K) - third_div)

    # trace-free shift gradient: with db[k][k] less div/3 the terms
    # -2/3 gt_ij div and -2/3 At_ij div are part of the products below
    def db(k, i):
        return dbeta(k, i) - third_div if k == i else dbeta(k, i)

    two_alpha = 2.0 * alpha
    for m, (i, j) in enumerate(PAIRS):
        s = adv(GT + m) - two_alpha * At[i, j]
        if i == j:
            s = s + 2.0 * (gt[i, 0] * db(j, 0) + gt[i, 1] * db(j, 1) + gt[i, 2] * db(j, 2))
        else:
            for k in range(3):
                s = s + gt[i, k] * db(j, k) + gt[j, k] * db(i, k)
        out[GT + m] = s
    kk = alpha * (AA + (1.0 / 3.0) * K * K)
    if have_matter:
        kk = kk + (4.0 * pi) * alpha * (rhoH + Str)
    out[TRK] = adv(TRK) - lap_a + kk
    X = []
    a8 = (8.0 * pi) * alpha
    for m, (i, j) in enumerate(PAIRS):
        x = half_alpha * Ric2[m] + ah * dd(CHI, i, j) - dd(ALP, i, j) + Gu_v[m]
        x = x - 2.0 * (hchi[i] * wal[i]) if i == j else x - hchi[i] * wal[j] - hchi[j] * wal[i]
        if have_matter:
            x = x - a8 * Sl[m]
        X.append(x)
    ctrX = chi * ((1.0 / 3.0) * contract_sym(gu2, Sym(X)))
    # At_ik (d_j beta^k - alpha At^k_j) + (i <-> j) + alpha K At_ij, the last as
    # (alpha K/2) delta^k_j in the bracket
    hak = half_alpha * K
    W = [[(db(j, k) + hak if j == k else db(j, k)) - alpha * Aud[k][j] for j in range(3)] for k in range(3)]
    for m, (i, j) in enumerate(PAIRS):
        s = adv(AT + m) + chi * X[m] - gt[i, j] * ctrX
        if i == j:
            s = s + 2.0 * (At[i, 0] * W[0][j] + At[i, 1] * W[1][j] + At[i, 2] * W[2][j])
        else:
            for k in range(3):
                s = s + At[i, k] * W[k][j] + At[j, k] * W[k][i]
        out[AT + m] = s
    # gt^ij y_j and -2 At^ij z_j collect the terms of d_t Gt^i that one tensor multiplies
    a43 = c43 * alpha
    a16 = (16.0 * pi) * alpha
    y, z = [], []
    az = 1.5 * (alpha * ichi)
    for j in range(3):
        ddivb = dd(BET + 0, j, 0) + dd(BET + 1, j, 1) + dd(BET + 2, j, 2)  # d_j d_k beta^k
        t = (1.0 / 3.0) * ddivb - a43 * dK[j]
        if have_matter:
            t = t - a16 * Jl[j]
        y.append(t)
        z.append(dal[j] + az * dchi[j])
    Gt_src = []  # d_t Gt^i without its advection
    for i in range(3):
        s = contract_sym(gu2, Sym([dd(BET + i, a, b) for (a, b) in PAIRS]))
        s = s + gu[i, 0] * y[0] + gu[i, 1] * y[1] + gu[i, 2] * y[2]
        s = s - (Gd[0] * db(0, i) + Gd[1] * db(1, i) + Gd[2] * db(2, i)) + Gd[i] * third_div
        s = s - 2.0 * (Atu[i, 0] * z[0] + Atu[i, 1] * z[1] + Atu[i, 2] * z[2])
        s = s + two_alpha * GA[i]
        Gt_src.append(s)
        out[GAM + i] = adv(GAM + i) + s
    out[ALP] = adv(ALP) - alpha * (c1 + c2 * alpha) * (g.input("kdiff") if split else K - Kref)
    for i in range(3):
        if split:  # m of beta^i and B^i has the switch on its advection
            out[BET + i] = adv(BET + i) + shift_on * (c75 * B[i])
            out[BB + i] = adv(BB + i) + shift_on * (Gt_src[i] - eta * B[i])
        else:
            out[BET + i] = shift_on * (adv(BET + i) + 0.75 * B[i])
            out[BB + i] = shift_on * (adv(BB + i) + Gt_src[i] - eta * B[i])
    if fluid:
        q = 24
        E, J, wJ, isg, P, iEP = fl["E"], fl["J"], fl["wJ"], fl["isg"], fl["P"], fl["iEP"]
        Str_f = fl["Str"]  # S^ij gamma_ij = S^ij gt_ij / chi
        # S^ij = chi^2 gt^ik gt^jl S_kl = chi^2 J^i J^j/(E + P) + chi P gt^ij (J^i = gt^ij J_j here)
        c2q = chi * chi * iEP
        cP = chi * P
        wq = [c2q * wJ[i] for i in range(3)]
        Su2 = [wq[i] * wJ[j] + cP * gu[i, j] if i == j else 2.0 * (wq[i] * wJ[j] + cP * gu[i, j])
               for (i, j) in PAIRS]
        # K_ij S^ij with K_ij = (At_ij + gt_ij K / 3)/chi
        KS = ichi * contract_sym(Su2, At) + (1.0 / 3.0) * K * Str_f
        Jda = chi * (wJ[0] * dal[0] + wJ[1] * dal[1] + wJ[2] * dal[2])  # J^j d_j alpha
        out[q] = isg * (alpha * KS - Jda)
        for i in range(3):
            s = (J[0] * dbeta(i, 0) + J[1] * dbeta(i, 1) + J[2] * dbeta(i, 2)) - E * dal[i]
            # S^jk d_i gamma_jk, gamma_jk = gt_jk / chi
            Sdg = contract_sym(Su2, Sym([dgt(i, a, b) for (a, b) in PAIRS]))
            cut.append(Sdg)
            s = s + half_alpha * (ichi * (Sdg - dchi[i] * Str_f))
            out[q + 1 + i] = isg * s
    if scalar:
        s = 24 + 4 * fluid
        Pi_ = u[s + 1]
        ddphi = contract_sym(gu2, Sym([dd(s, a, b) for (a, b) in PAIRS]))
        Gd_dphi = Gd[0] * dphi[0] + Gd[1] * dphi[1] + Gd[2] * dphi[2]
        wchi_dphi = wchi[0] * dphi[0] + wchi[1] * dphi[1] + wchi[2] * dphi[2]
        lap_phi = chi * (ddphi - Gd_dphi) - 0.5 * wchi_dphi
        da_dphi = chi * (wphi[0] * dal[0] + wphi[1] * dal[1] + wphi[2] * dal[2])
        out[s] = adv(s) - alpha * Pi_
        out[s + 1] = adv(s + 1) + alpha * (K * Pi_ - lap_phi) - da_dphi
    if split:
        S = split_layout(fluid, scalar)
        g.cut = cut + Ric2 + Gd + [x for t in Gu for x in t.c] + gu.c
        if S["early"]:
            g.cut += [x for row in Aud for x in row] + Atu.c + GA + [AA]
        return g, S, out
    # ---- constraints (diagnostic outputs, same graph) ----
    #  H   = R + 2/3 K^2 - At_ij At^ij - 16 pi rho_H,   R = chi gt^ij R_ij
    #  M^i = gt^ik gt^jl Dt_j At_kl - 3/(2 chi) At^ij d_j chi - 2/3 gt^ij d_j K - 8 pi gt^ij J_j
    #  with R = 1/2 chi gt^ij 2R~_ij + 2 gt^ij D_i D_j chi - 5/(2 chi) gt^ij d_i chi d_j chi,
    #  and gt^jl Dt_j At_kl = gt^jl d_j At_kl - At^j_m Gamma^m_jk - Gd^m At_km
    dchi2 = wchi[0] * dchi[0] + wchi[1] * dchi[1] + wchi[2] * dchi[2]
    trDD = (contract_sym(gu2, Sym([dd(CHI, i, j) for (i, j) in PAIRS]))
            - (Gd[0] * dchi[0] + Gd[1] * dchi[1] + Gd[2] * dchi[2]))
    H = (0.5 * chi) * contract_sym(gu2, Sym(Ric2)) + 2.0 * trDD - 2.5 * ichi * dchi2 + (2.0 / 3.0) * K * K - AA
    if have_matter:
        H = H - (16.0 * pi) * rhoH
    Y = []
    for k in range(3):
        s = None
        for j in range(3):
            for l in range(3):
                t = gu[j, l] * dAt(j, k, l)
                s = t if s is None else s + t
        for j in range(3):
            for m in range(3):
                s = s - Aud[j][m] * Gu[m][j, k]
        s = s - Gd[0] * At[k, 0] - Gd[1] * At[k, 1] - Gd[2] * At[k, 2] - (2.0 / 3.0) * dK[k]
        if have_matter:
            s = s - (8.0 * pi) * Jl[k]
        Y.append(s)
    m15 = 1.5 * ichi
    M = []
    for i in range(3):
        Adchi = Atu[i, 0] * dchi[0] + Atu[i, 1] * dchi[1] + Atu[i, 2] * dchi[2]
        M.append((gu[i, 0] * Y[0] + gu[i, 1] * Y[1] + gu[i, 2] * Y[2]) - m15 * Adchi)
    g.constraints = [H] + M
    return g, L, out
