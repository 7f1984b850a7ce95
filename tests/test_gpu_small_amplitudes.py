"""Amplitudes far below a column's norm, as the first step from unit columns
makes them (one empty orbital's amplitude is dt times a coupling): their own
accuracy, not that of the column, against the exponential of the context's
generator in extended precision (FP64) and against FP64 (mixed)."""
import math

import numpy as np
import pytest

import iesh_inputs as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


def _step(P, md, n, x, p, dt, precision, **kw):
    occ = np.repeat((md["M"] // 2 - md["Ne"] // 2 + np.arange(md["Ne"]))[None], n, 0).astype(np.int16)
    ctx = P.Context(md, n, precision=precision, norm_tol=-1.0, **kw)
    ctx.set_state(x, p, occ, W.unit_coefficients(occ, md["M"] + 1).astype(ctx.cdtype))
    lam0, q0, _ = ctx.eigen()
    ctx.run(dt, 1, seed=2)
    lam1, q1, _ = ctx.eigen()
    st, K = ctx.get_state(), ctx.propagator_terms()
    assert np.array_equal(st["occ"], occ)
    g = ctx.hop_probabilities(dt)
    ctx.close()
    return st, K, occ, (lam0, q0, lam1, q1), g


def _generator(md, lam0, q0, v0, lam1, q1, v1, dt):
    """L and W of H = L - i W from the context's eigenpairs (the double well's
    coupling does not depend on x), in extended precision."""
    dh = -np.longdouble(md["mass"]) * md["par"][0] ** 2 * md["par"][1]
    Wm = 0
    for lam, q, v in ((lam0, q0, v0), (lam1, q1, v1)):
        lam, q = lam.astype(np.longdouble), q.astype(np.longdouble)
        gap = lam[None, :] - lam[:, None]
        np.fill_diagonal(gap, np.inf)
        Wm = Wm + np.longdouble(0.5 * dt) * v * dh * np.outer(q, q) / gap
    return np.longdouble(0.5 * dt) * (lam0.astype(np.longdouble) + lam1), Wm


def _exponential(L, Wm, cols):
    """exp(-i H) on unit columns: a Taylor series in extended precision."""
    C = np.zeros((len(L), len(cols)), np.clongdouble)
    C[cols, np.arange(len(cols))] = 1
    c = 0.5 * (L.max() + L.min())
    out, term = C.copy(), C
    for k in range(1, 60):
        term = (-1j * (L - c)[:, None] * term - Wm @ term) / k
        out = out + term
    return out * np.exp(np.clongdouble(-1j) * c)


# The unit of an entry that starts from zero is at most grow 2^-60 (grow: what
# an entry may gain in K orders), each of K orders rounds it within 4 units at
# random, and leaves out products of 2^-46.5 of the largest coupling, a quarter
# of that on average
@pytest.mark.parametrize("M,Ne", [(40, 20), (100, 50), (200, 30)])
@pytest.mark.parametrize("deflation", [False, True])
@pytest.mark.parametrize("v", [2e-3, 2e-4, 2e-6])
def test_fp64(P, M, Ne, deflation, v):
    md, dt, n = W.double_well(M, Ne), 1.0, 2
    x, p = np.array([0.3, -1.0]), np.array([v, -v]) * md["mass"]
    st, K, occ, e, _ = _step(P, md, n, x, p, dt, P.PREC_FP64, deflation=deflation)
    empty = np.setdiff1d(np.arange(M + 1), occ[0])
    for t in range(n):
        L, Wm = _generator(md, e[0][t], e[1][t], p[t] / md["mass"], e[2][t], e[3][t], st["p"][t] / md["mass"], dt)
        ref = _exponential(L, Wm, occ[t])
        disc = L + np.abs(Wm).sum(1)
        rho = 0.5 * float((disc[:-1].max() if deflation else disc.max()) - L.min())
        w, k = 2.0 / rho * float(np.abs(Wm).max()), int(K[t])
        grow = 1.3 * w * math.sqrt(M + 1) * k * (k + 1)
        err = np.abs(st["C"][t].T - ref)[empty].astype(np.float64)
        unit = max(grow * 2.0 ** -60, 2.0 ** -76)
        assert np.sqrt((err ** 2).mean()) <= k * (4 * unit + max(w, 2.0 ** -26) * 2.0 ** -48)


# FP32 products and sums: a handful of roundings of 2^-24 per amplitude
# (couplings 3, the product 1 and its digits 1, K orders and phases), and the
# hop probability has two such factors
@pytest.mark.parametrize("M,Ne", [(140, 30), (200, 100), (255, 9)])
@pytest.mark.parametrize("v", [2e-3, 2e-5])
def test_mixed(P, M, Ne, v):
    md, dt, n = W.double_well(M, Ne), 1.0, 4
    x, p = np.array([0.3, -1.0, 0.0, 1.0]), np.array([v, -v, 0.5 * v, 3 * v]) * md["mass"]
    a, _, occ, _, ga = _step(P, md, n, x, p, dt, P.PREC_FP64)
    b, K, _, _, gb = _step(P, md, n, x, p, dt, P.PREC_MIXED)
    empty = np.setdiff1d(np.arange(M + 1), occ[0])
    for t in range(n):
        ca, cb = a["C"][t][:, empty], b["C"][t][:, empty]
        units = (6 + K[t]) * 2.0 ** -24
        assert np.abs(ca - cb).max() <= 2 * units * np.abs(ca).max()
        assert np.sqrt((np.abs(ca - cb) ** 2).mean()) <= units * np.sqrt((np.abs(ca) ** 2).mean())
        assert np.abs(ga[t] - gb[t]).max() <= 4 * units * ga[t].max()
