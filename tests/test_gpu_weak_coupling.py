"""Roots of the secular equation for couplings far below the level spacing (an
adsorbate far from the surface): the eigenvector components against first-order
perturbation theory, which is exact to (coupling / spacing)^2."""
import numpy as np
import pytest

import iesh_inputs as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


def _components(P, gamma, precision):
    """Impurity components of all bath-like orbitals but the two outermost
    (whose interval closes on the pole at these couplings), of a cold start and
    after two steps, with the level at gap middles; the components by
    perturbation theory, z_k / |eps_k - h|."""
    md = W.double_well(50)
    md["Gamma"] = gamma
    ctx = P.Context(md, 8, precision=precision)
    eps, z = ctx.bath()
    k = np.array([5, 11, 17, 23, 24, 30, 37, 44])
    a = md["mass"] * md["par"][0] ** 2
    level = lambda x: 0.5 * a * (md["par"][1] ** 2 - 2 * md["par"][1] * x) + md["par"][2]
    x = (level(0.0) - 0.5 * (eps[k] + eps[k + 1])) / (a * md["par"][1])
    occ = W.lowest_occupations(8, md["Ne"])
    ctx.set_state(x, np.full(8, 1e-3), occ, W.unit_coefficients(occ, 51).astype(ctx.cdtype))
    for step in range(2):
        if step:
            ctx.run(1.0, 2, seed=1)
        st = ctx.get_state()
        lam, q0, F = ctx.eigen()
        assert np.all(np.isfinite(F)) and np.all(st["status"] == 0)
        for t in range(8):
            h = level(st["x"][t])
            imp = int(np.abs(lam[t] - h).argmin())
            assert abs(q0[t, imp] - 1.0) < 1e-15
            bath = np.delete(q0[t], imp)
            yield bath[1:-1], (np.abs(z / (eps - h)))[1:-1]
    ctx.close()


# The roots are resolved to 8 units of 2^-53 (mixed: 2^-44) of the secular
# function's terms, two of which are of the size of the level's distance to the
# pole; h and the poles carry 2^-53 of the band over half a spacing (10^-13).
# z^2 from 10^-20 down: its second derivative, spacing^3 / z^4, leaves FP32
@pytest.mark.parametrize("gamma", [1e-18, 1e-24, 1e-40])
@pytest.mark.parametrize("prec,tol", [("PREC_FP64", 1e-12), ("PREC_MIXED", 4e-12)])
def test_components(P, gamma, prec, tol):
    for got, ref in _components(P, gamma, getattr(P, prec)):
        assert np.abs(got / ref - 1.0).max() < tol


def test_occupied_energy(P):
    """Couplings of 10^-11 and 10^-16: the energy is the sum of the lowest
    uncoupled levels and its gradient the occupied adsorbate levels'."""
    import torch
    from paper_2212_00518_gb300 import eocc as E
    for scale in (1e-11, 1e-16):
        wl = W.eocc_workload(M=60, B=64)
        wl["Vbar"] = wl["Vbar"] * scale
        x = torch.from_numpy(wl["x"]).cuda().requires_grad_(True)
        th = torch.from_numpy(wl["theta"]).cuda()
        en = E.eocc(x, th, E.EOccModel(wl))
        dx, = torch.autograd.grad(en.sum(), x)
        nodes, _ = np.polynomial.legendre.leggauss(30)
        eps = np.concatenate([0.25 * nodes - 0.25, 0.25 * nodes + 0.25])
        g = wl["theta"][2:14].reshape(2, 6)
        for b in range(64):
            h = wl["theta"][:2] + g @ wl["x"][b]
            lev = np.concatenate([eps, h])
            occ = np.sort(np.argsort(lev)[:wl["Ne"]])
            assert abs(en[b].item() - lev[occ].sum()) < 1e-13 * np.abs(lev).sum()
            ref = g[[i - 60 for i in occ if i >= 60]].sum(0)
            assert np.abs(dx[b].detach().cpu().numpy() - ref).max() < 1e-9
