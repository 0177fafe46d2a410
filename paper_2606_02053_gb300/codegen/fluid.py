"""Fluid pieces of the right-hand side in the expression DSL.

Perfect fluid with P = w rho (section "Physical system settings"), evolved in
conservative 3+1 form (tau~ = sqrt(gamma) E, S~_i = sqrt(gamma) J_i) with the
Kurganov-Tadmor central scheme (the paper's fluid method):

* ``prim``: cell-centred recovery of (rho, v_i) from (tau~, S~_i).  With
  h W^2 = (1 + w) rho W^2:  E = h W^2 - w rho,  J_i = h W^2 v_i, hence
  w rho^2 + (1 - w) E rho + (J^2 - E^2) = 0 and rho is its positive root.
* ``face_flux(d)``: numerical flux through the face between cells c and
  c + e_d: minmod-limited linear reconstruction of (rho, v_i) from cells
  c-1 .. c+2, face metric = mean of the two adjacent cells, and
  H = (F(q_L) + F(q_R))/2 - a (U(q_R) - U(q_L))/2 with a the largest
  |characteristic speed| of both states, speeds
  lambda_pm = alpha/(1 - v^2 w) [v^d (1 - w) pm sqrt(w (1 - v^2)(gamma^dd (1 - v^2 w) - v^d v^d (1 - w)))] - beta^d.
"""
from __future__ import annotations

from .expr import Graph, fabs, fmax, minmod, mulr, sqrt

PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
PIDX = {(0, 0): 0, (0, 1): 1, (0, 2): 2, (1, 0): 1, (1, 1): 3, (1, 2): 4, (2, 0): 2, (2, 1): 4, (2, 2): 5}


def _cofactors(gt):
    """Cofactors of a symmetric matrix (the inverse times the determinant) and the determinant."""
    c = [gt[3] * gt[5] - gt[4] * gt[4], gt[2] * gt[4] - gt[1] * gt[5], gt[1] * gt[4] - gt[2] * gt[3],
         gt[0] * gt[5] - gt[2] * gt[2], gt[1] * gt[2] - gt[0] * gt[4], gt[0] * gt[3] - gt[1] * gt[1]]
    return c, gt[0] * c[0] + gt[1] * c[1] + gt[2] * c[2]


def _row(c, i, v):
    return c[PIDX[(i, 0)]] * v[0] + c[PIDX[(i, 1)]] * v[1] + c[PIDX[(i, 2)]] * v[2]


def _square(c, v):
    """sum_ij c_ij v_i v_j"""
    return v[0] * _row(c, 0, v) + v[1] * _row(c, 1, v) + v[2] * _row(c, 2, v)


def prim():
    """Inputs: chi, gt[6], tau, S[3]  ->  outputs rho, v_0, v_1, v_2.

    The recovery is homogeneous in (E, J_i, rho), so it is done with the
    densitised tau, S_i (E = chi^{3/2} tau, J_i = chi^{3/2} S_i) and the factor
    chi^{3/2} goes on rho alone: v_i = S_i / (tau + w rho~), rho = chi^{3/2} rho~."""
    g = Graph()
    names = ["chi"] + [f"gt{m}" for m in range(6)] + ["tau", "S0", "S1", "S2"]
    x = {n: g.input(n) for n in names}
    w = g.param("w")
    chi, tau = x["chi"], x["tau"]
    S = [x[f"S{i}"] for i in range(3)]
    c, det = _cofactors([x[f"gt{m}"] for m in range(6)])
    k = chi * det.rcp()  # gamma^ij = k c_ij
    D = tau * tau - k * _square(c, S)
    a = (1.0 - w) * tau
    # positive root, rationalised to avoid cancellation: 2 (E^2 - J^2) / (a + sqrt(a^2 + 4 w (E^2 - J^2)))
    rho = 2.0 * D * (a + sqrt(a * a + (4.0 * w) * D)).rcp()
    iEP = (tau + w * rho).rcp()
    out = [chi * sqrt(chi) * rho] + [S[i] * iEP for i in range(3)]
    return g, names, out


def face_flux(d: int):
    """Inputs: rho/v at cells c-1..c+2 (q{o}_{m}, o = 0..3, m = rho, v0..2) and
    metric at cells c, c+1 (chi{s}, alpha{s}, beta{s} (component d), gt{s}_{m}).
    Outputs: H_tau, H_S0, H_S1, H_S2.

    The kernel is bound by the FP64 pipe.  The face metric is kept doubled (the
    sum of both cells: lapse, shift and speeds then carry a factor 2, the flux
    a factor 1/4), the inverse metric is never formed (gamma^ij = k c_ij with the
    cofactors c_ij of the doubled metric), reciprocals come in pairs from one
    division, and with s = alpha v^d - beta the fluxes are F_E = E s + alpha P v^d,
    F_i = J_i s + alpha P delta_id.  The two speeds of a side, (A +- R) - beta,
    have the largest modulus |A - beta| + |R| (R has the sign of the lapse).  A flux is antisymmetric
    bitwise under the exchange of its sides (with the odd components negated):
    what the sides contribute meets only in sums of two rounded terms (mulr)."""
    g = Graph()
    names = [f"q{o}_{m}" for o in range(4) for m in range(4)]
    for s in range(2):
        names += [f"chi{s}", f"alpha{s}", f"beta{s}"] + [f"gt{s}_{m}" for m in range(6)]
    x = {n: g.input(n) for n in names}
    w, sqw = g.param("w"), g.param("sqrt_w")
    omw, opw = 1.0 - w, 1.0 + w
    q = [[x[f"q{o}_{m}"] for m in range(4)] for o in range(4)]
    qL = [q[1][m] + 0.5 * minmod(q[1][m] - q[0][m], q[2][m] - q[1][m]) for m in range(4)]
    qR = [q[2][m] - 0.5 * minmod(q[2][m] - q[1][m], q[3][m] - q[2][m]) for m in range(4)]
    chi2 = x["chi0"] + x["chi1"]
    alpha2 = x["alpha0"] + x["alpha1"]
    beta2 = x["beta0"] + x["beta1"]
    c, det = _cofactors([x[f"gt0_{m}"] + x[f"gt1_{m}"] for m in range(6)])
    chi = 0.5 * chi2
    c32 = chi * sqrt(chi)
    r = (det * c32).rcp()
    k = chi2 * (c32 * r)  # gamma^ij = k c_ij
    hs = 0.25 * (det * r)  # sqrt(gamma)/2, and 1/2 for the doubled lapse and shift
    wk = w * k
    gdd = k * c[PIDX[(d, d)]]
    aw = w * alpha2
    U, F, speed = [], [], []
    for side in (qL, qR):
        rho, v = side[0], side[1:]
        vd = k * _row(c, d, v)
        vv = _square(c, v)
        one_v2 = 1.0 - k * vv
        one_wv2 = 1.0 - wk * vv
        pair = (one_v2 * one_wv2).rcp()
        hW2 = (opw * rho) * (pair * one_wv2)
        pre = alpha2 * (pair * one_v2)
        E = hW2 - w * rho
        J = [hW2 * v[i] for i in range(3)]
        U.append([E] + J)
        s = alpha2 * vd - beta2
        aP = aw * rho
        F.append([E * s + aP * vd] + [J[i] * s + aP if i == d else mulr(J[i], s) for i in range(3)])
        disc = one_v2 * (gdd * one_wv2 - omw * (vd * vd))
        speed.append(fabs((pre * omw) * vd - beta2) + fabs(pre * sqw) * sqrt(disc))
    a = fmax(speed[0], speed[1])
    out = [hs * ((F[0][m] + F[1][m]) - a * (U[1][m] - U[0][m])) for m in range(4)]
    return g, names, out
