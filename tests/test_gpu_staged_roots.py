"""Roots of the secular equation found in stages (FP32 and double-float sums
before one FP64 evaluation): eigenpairs of small batches against LAPACK where
a stage decides narrowly -- roots at the middle of a pole gap, a level on a
bath energy, vanishing and strong couplings -- from cold and warm starts."""
import numpy as np
import pytest

import iesh_inputs as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


def _dense(md, eps, z, x):
    k = md["mass"] * md["par"][0] ** 2
    g = md["par"][1]
    h = 0.5 * k * (g * g - 2 * g * x) + md["par"][2]
    H = np.diag(np.concatenate([[h], eps]))
    H[0, 1:] = H[1:, 0] = z
    return H


def _level_to_x(md, h):
    """Position where the impurity level is h."""
    k = md["mass"] * md["par"][0] ** 2
    g = md["par"][1]
    return (0.5 * k * g * g + md["par"][2] - h) / (k * g)


@pytest.mark.parametrize("M,gamma", [(2, 3e-3), (9, 1e-12), (40, 6.4e-3), (100, 3e-3), (100, 2.0), (255, 1e-6)])
def test_eigenpairs_at_narrow_decisions(P, M, gamma):
    """Levels on bath energies, at gap middles and beside them: eigenvalues to
    a few 2^-53 of the spectrum (both sides' backward errors), the impurity
    weights q0^2 to their conditioning by the nearest other eigenvalue."""
    md = W.double_well_paper(40)
    md.update(M=M, Ne=min(112, max(1, M // 2)), Gamma=gamma)
    ctx = P.Context(md, 64)
    eps, z = ctx.bath()
    rng = np.random.default_rng(M)
    k = rng.integers(0, max(M - 1, 1), 10)
    mids = 0.5 * (eps[k] + eps[np.minimum(k + 1, M - 1)])
    levels = np.concatenate([eps[k], mids, mids * (1 + 1e-7), mids * (1 - 1e-13), rng.uniform(-0.05, 0.05, 24)])
    x = np.array([_level_to_x(md, h) for h in levels])
    n = x.size
    occ = W.lowest_occupations(n, md["Ne"])
    C = W.unit_coefficients(occ, M + 1)
    for step in range(2):  # cold, then warm after a step
        if step == 0:
            ctx.set_state(x, np.full(n, 0.3), occ, C)
        else:
            ctx.run(10.0, 1, seed=1)
        xs = ctx.get_state()["x"]
        lam, q0, _ = ctx.eigen()
        for t in range(n):
            H = _dense(md, eps, z, xs[t])
            ev, Q = np.linalg.eigh(H)
            scale = np.abs(ev).max()
            assert np.abs(lam[t] - ev).max() <= 2e-14 * scale
            gap = np.minimum(np.diff(ev, prepend=-1e9), np.diff(ev, append=1e9))
            assert np.all(np.abs(q0[t] ** 2 - Q[0] ** 2) <= 1e-13 + 1e-14 * scale / gap)
    assert np.all(ctx.get_state()["status"] == 0)
    ctx.close()


def test_occupied_energy_near_mid_gap(P):
    """E_occ and its gradients over many geometries against a plain 64-bit
    bisection of the same secular equation, root by root in the largest
    error (a root lost at the middle of its gap showed up as 1e-10)."""
    import torch
    from paper_2212_00518_gb300 import eocc as E
    wl = W.eocc_workload(M=60, B=40000, seed=8)
    x = torch.from_numpy(wl["x"]).cuda()
    th = torch.from_numpy(wl["theta"]).cuda()
    m = E.EOccModel(wl)
    En, saved, st = m.forward(x, th)
    assert int(st.max()) == 0
    lo, hi = wl["band"]
    xg, wg = np.polynomial.legendre.leggauss(30)
    eps = np.concatenate([0.5 * (0 - lo) * xg + 0.5 * lo, 0.5 * hi * xg + 0.5 * hi])
    w = np.concatenate([0.5 * (0 - lo) * wg, 0.5 * hi * wg])
    n = 3000
    X = wl["x"][:n]
    h = np.stack([wl["theta"][0] + X @ wl["theta"][2:8], wl["theta"][1] + X @ wl["theta"][8:14]], 1)
    d = X - wl["R"]
    c = wl["Vbar"] * np.exp(-0.5 * np.stack([(d[:, :3] ** 2).sum(1), (d[:, 3:] ** 2).sum(1)], 1) / wl["theta"][14:] ** 2)
    H = np.zeros((n, 62, 62))
    H[:, 0, 0], H[:, 1, 1] = h[:, 0], h[:, 1]
    H[:, np.arange(2, 62), np.arange(2, 62)] = eps
    for a in range(2):
        H[:, a, 2:] = H[:, 2:, a] = c[:, a, None] * np.sqrt(w)
    ev, Q = np.linalg.eigh(H)
    Ne = wl["Ne"]
    # 31 roots of magnitude below 1, LAPACK's backward error a few n 2^-53
    assert np.abs(En.cpu().numpy()[:n] - ev[:, :Ne].sum(1)).max() <= 62 * 31 * 2.0 ** -53
    for a in range(2):
        S = (Q[:, a, :Ne] ** 2).sum(1)
        gap = ev[:, Ne] - ev[:, Ne - 1]  # rotations among the occupied leave the sum
        assert np.all(np.abs(saved[:n, a].cpu().numpy() - S) <= 1e-12 + 62 * 2.0 ** -53 / gap)
