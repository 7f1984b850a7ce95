"""Propagation with the top level deflated, where what rounding leaves of a
column along that level grows with the Chebyshev polynomials: the tensor-core
kernels' number ranges (FP16 digits, 64-bit fixed point) against the oracle."""
import functools

import numpy as np
import pytest

import iesh_inputs as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


X, V = np.array([-2.0, -2.0, 0.0, 0.0, 0.0, 2.0]), np.array([0.002, 1.0, 0.002, 0.2, 1.0, 0.2])


@functools.lru_cache(maxsize=None)
def _case(M, Ne, dt):
    """A column in the top level with a phase, one with equal entries, generic
    ones, and the oracle's step of them."""
    md = W.double_well(M, Ne)
    n, N = len(X), M + 1
    occ = W.random_occupations(n, N, Ne, 3)
    C = W.mixed_coefficients(occ, N, 4, 0.5)
    C[:, 0] = 0.0
    C[:, 0, N - 1] = np.exp(1j * (0.3 + np.arange(n)))
    C[:, 1] = np.exp(1j * np.arange(N)) / np.sqrt(N)
    B = O.bind(md)
    ref = [O.step_one(B, X[t], V[t] * md["mass"], occ[t].astype(np.int32), C[t].T, dt, seed=5, traj=t, n=0)["C"]
           for t in range(n)]
    return md, occ, C, ref


def _check(P, M, Ne, dt, precision, tol, bound):
    md, occ, C, ref = _case(M, Ne, dt)
    ctx = P.Context(md, len(X), precision=precision, prop_tol=tol, norm_tol=-1.0)
    ctx.set_state(X, V * md["mass"], occ, C.astype(ctx.cdtype))
    ctx.run(dt, 1, seed=5)
    st = ctx.get_state()
    K = ctx.propagator_terms()
    ctx.close()
    assert np.all(np.isfinite(st["C"]))
    for t in range(len(X)):
        assert np.abs(st["C"][t].T - ref[t]).max() <= bound(K[t])


# each order rounds a few results (2^-24) and carries them k-fold, those along
# the deflated level at most 16-fold: (2 K (K + 1) + 32 (K + 1) + 16) 2^-24
@pytest.mark.parametrize("M,Ne", [(128, 16), (200, 20), (191, 9)])
@pytest.mark.parametrize("dt", [1.0, 1.5])
@pytest.mark.parametrize("tol", [0.0, 1e-10, 1e-12])
def test_mixed(P, M, Ne, dt, tol):
    _check(P, M, Ne, dt, P.PREC_MIXED, tol,
           lambda K: (2.0 * K * (K + 1) + 32 * (K + 1) + 16) * 2.0 ** -24)


# as above with 2^-53 and the deflated level's 10^3; the oracle's generator
# carries 10^-12 from its own eigensolver
@pytest.mark.parametrize("M,Ne", [(40, 20), (100, 50), (200, 12)])
@pytest.mark.parametrize("dt", [1.5, 3.0, 3.4, 4.0])
def test_fp64(P, M, Ne, dt):
    _check(P, M, Ne, dt, P.PREC_FP64, 0.0,
           lambda K: 1e-12 + (2.0 * K * (K + 1) + 2e3 * (K + 1)) * 2.0 ** -53)
