"""Amplitudes far below a column's norm, as the first step from unit columns
makes them (one empty orbital's amplitude is dt times a coupling): their own
accuracy, not that of the column: mixed precision against FP64."""
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
    ctx.run(dt, 1, seed=2)
    st, K = ctx.get_state(), ctx.propagator_terms()
    assert np.array_equal(st["occ"], occ)
    g = ctx.hop_probabilities(dt)
    ctx.close()
    return st, K, occ, g


# FP32 products and sums: a handful of roundings of 2^-24 per amplitude
# (couplings 3, the product 1 and its digits 1, K orders and phases), and the
# hop probability has two such factors
@pytest.mark.parametrize("M,Ne", [(140, 30), (200, 100), (255, 9)])
@pytest.mark.parametrize("v", [2e-3, 2e-5])
def test_mixed(P, M, Ne, v):
    md, dt, n = W.double_well(M, Ne), 1.0, 4
    x, p = np.array([0.3, -1.0, 0.0, 1.0]), np.array([v, -v, 0.5 * v, 3 * v]) * md["mass"]
    a, _, occ, ga = _step(P, md, n, x, p, dt, P.PREC_FP64)
    b, K, _, gb = _step(P, md, n, x, p, dt, P.PREC_MIXED)
    empty = np.setdiff1d(np.arange(M + 1), occ[0])
    for t in range(n):
        ca, cb = a["C"][t][:, empty], b["C"][t][:, empty]
        units = (6 + K[t]) * 2.0 ** -24
        assert np.abs(ca - cb).max() <= 2 * units * np.abs(ca).max()
        assert np.sqrt((np.abs(ca - cb) ** 2).mean()) <= units * np.sqrt((np.abs(ca) ** 2).mean())
        assert np.abs(ga[t] - gb[t]).max() <= 4 * units * ga[t].max()
