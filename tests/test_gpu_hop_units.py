"""Units of the FP64 hop ratios in fixed point (csrc/iesh_hop_fx.cuh): every
electron's column has its own, small pivots do not multiply a row's rounding."""
import numpy as np
import pytest

import iesh_inputs as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


def _probs(P, md, x, p, occ, C):
    ctx = P.Context(md, x.shape[0], norm_tol=-1.0)
    ctx.set_state(x, p, occ, C)
    g = ctx.hop_probabilities(100.0)
    ctx.close()
    return g


# determinant ratios do not change with an electron's scale, and powers of two
# round nothing: the same bits at every position of the scaled column
@pytest.mark.parametrize("M,Ne,weight", [(40, 20, 0.3), (24, 7, 0.3), (100, 50, 0.9), (150, 112, 0.5)])
def test_scaled_electrons_same_bits(P, M, Ne, weight):
    md = W.double_well_paper(40)
    md.update(M=M, Ne=Ne)
    N, shifts = M + 1, (-8, -16, -24, -60, 30, None)
    n = 1 + Ne * len(shifts)
    x, p = W.thermal_harmonic(1, md["mass"], md["par"][0], 5 * 9.5e-4, M)
    occ = W.random_occupations(1, N, Ne, M + 1)
    C = np.repeat(W.mixed_coefficients(occ, N, M + 2, weight), n, 0)
    for a in range(Ne):
        for i, sh in enumerate(shifts):
            t = 1 + a * len(shifts) + i
            if sh is None:  # every column, from 2^-30 to 2^30
                C[t] *= np.ldexp(1.0, (np.arange(Ne) * 13 + a) % 61 - 30)[:, None]
            else:
                C[t, a] *= 2.0 ** sh
    g = _probs(P, md, np.repeat(x, n), np.repeat(p, n), np.repeat(occ, n, 0), C)
    assert g[0].max() > 0
    assert np.array_equal(g, np.broadcast_to(g[0], g.shape))


def _ratios(S, Cu):
    """C_u S^{-1} by Gaussian elimination in extended precision."""
    A, B = S.astype(np.clongdouble).T.copy(), Cu.astype(np.clongdouble).T.copy()
    n = len(A)
    for k in range(n):
        j = k + int(np.abs(A[k:, k]).argmax())
        A[[k, j]], B[[k, j]] = A[[j, k]], B[[j, k]]
        f = A[k + 1:, k] / A[k, k]
        A[k + 1:, k:] -= np.outer(f, A[k, k:])
        B[k + 1:] -= np.outer(f, B[k])
    for k in range(n - 1, -1, -1):
        B[k] = (B[k] - A[k, k + 1:] @ B[k + 1:]) / A[k, k]
    return B.T


def test_small_pivots(P):
    """One electron nearly out of the occupied orbitals, against ratios in
    extended precision; the couplings are taken from states whose ratios are 1
    and -1, so that nothing but the ratios is compared."""
    md = W.double_well_paper(40)
    N, Ne = 41, 20
    md.update(M=40, Ne=Ne)
    eps = [1e-2, 1e-3, 2e-4, 1e-6, 1e-12]
    n = 2 + len(eps)
    x, p = W.thermal_harmonic(1, md["mass"], md["par"][0], 5 * 9.5e-4, 3)
    occ = W.random_occupations(1, N, Ne, 5)
    o = np.sort(occ[0])
    un = np.setdiff1d(np.arange(N), o)
    C = np.repeat(W.mixed_coefficients(occ, N, 6, 0.3), n, 0)
    for t, sign in enumerate((1.0, -1.0)):
        C[t] = 0.0
        C[t][np.arange(Ne), o] = 1.0
        C[t][:, un] = sign
    for t, e in enumerate(eps):
        v = C[2 + t, -1]
        v[o] *= e
        v[un[0]] = 1.0
        v /= np.linalg.norm(v)
    g = _probs(P, md, np.repeat(x, n), np.repeat(p, n), np.repeat(occ, n, 0), C)
    k = (g[0] - g[1])[:, un].T  # -2 dt v d_{m, s_a}
    for t in range(len(eps)):
        Z = C[2 + t].T
        R = _ratios(Z[o], Z[un])
        ref = np.maximum(0.0, R.real.astype(np.float64) * k)
        # Ne roundings of the factors and of each substitution, growth 8
        tol = 3 * Ne * 8 * 2.0 ** -53 * np.abs(R).max(1, keepdims=True).astype(np.float64) * np.abs(k)
        assert np.all(np.abs(g[2 + t][:, un].T - ref) <= tol + 1e-300)
