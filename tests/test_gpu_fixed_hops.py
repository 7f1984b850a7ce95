"""Hop probabilities of the FP64 path with the substitutions in 64-bit fixed
point (csrc/iesh_hop_fx.cuh) against the oracle's determinant ratios: edges of
the quads and of the passes over unoccupied rows, and the calls that leave the
fixed-point range and take the FP64 substitution."""
import numpy as np
import pytest

import iesh_inputs as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


def _case(P, M, Ne, weight, change=None, n=4):
    md = W.double_well_paper(40)
    md.update(M=M, Ne=Ne)
    dt, N = 100.0, M + 1
    x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 5 * 9.5e-4, M)
    occ = W.random_occupations(n, N, Ne, M + 1)
    C = W.mixed_coefficients(occ, N, M + 2, weight)
    if change is not None:
        change(C, occ)
    ctx = P.Context(md, n, norm_tol=-1.0)
    ctx.set_state(x, p, occ, C)
    g = ctx.hop_probabilities(dt)
    ctx.close()
    B = O.bind(md)
    for t in range(n):
        d = O.eigen(B, x[t])[3]
        ref = O.hop_probs(occ[t], C[t].T, d, p[t] / md["mass"], dt)[0]
        S = C[t].T[occ[t]]
        cond = np.linalg.cond(S / np.abs(S).max(axis=1, keepdims=True))
        # the couplings come from two eigensolvers (1e-10 of the largest
        # probability), the ratios carry Ne roundings times the condition
        tol = 1e-10 + 2.0 ** -52 * Ne * cond
        assert np.abs(g[t] - ref).max() <= tol * max(np.abs(ref).max(), 1e-300)
    return g


# one electron, fewer than a quad, one past it, one unoccupied orbital, a short
# last quad of rows, rows past one pass (64 and 128), the largest Ne
@pytest.mark.parametrize("M,Ne", [(1, 1), (2, 2), (5, 3), (8, 5), (9, 9), (31, 16), (64, 1), (100, 37), (100, 36), (100, 50),
                                  (180, 52), (180, 51), (200, 100), (150, 112)])
@pytest.mark.parametrize("weight", [0.2, 0.8])
def test_hop_probabilities(P, M, Ne, weight):
    _case(P, M, Ne, weight)


# strongly mixed columns: entries of U1 past 1.75, column sums from 1 to past
# 15, rows that grow past the headroom and rows that do not
@pytest.mark.parametrize("M,Ne", [(17, 9), (24, 12), (40, 20), (100, 50), (200, 100)])
@pytest.mark.parametrize("weight", [0.9, 0.97, 1.0])
def test_strong_mixing(P, M, Ne, weight):
    _case(P, M, Ne, weight, n=12)


def test_rows_of_any_scale(P):
    """Each unoccupied row has its own unit: rows far below the others, far
    above them, and zero rows."""
    def change(C, occ):
        for t in range(C.shape[0]):
            un = [m for m in range(C.shape[2]) if m not in set(occ[t])]
            C[t][:, un[0]] = 0.0
            C[t][:, un[1]] *= 2.0 ** -200
            C[t][:, un[2]] *= 2.0 ** 40
    _case(P, 60, 30, 0.5, change)


@pytest.mark.parametrize("what", ["pivot", "growth", "nan"])
def test_outside_the_fixed_point_range(P, what):
    """Entries of U1 of 2 and more, rows that grow past the headroom: the FP64
    substitution; a NaN gives no probability above zero in its row."""
    def change(C, occ):
        for t in range(C.shape[0]):
            o = np.sort(occ[t])
            un = [m for m in range(C.shape[2]) if m not in set(o)]
            if what == "pivot":
                C[t][1:, o] *= 8.0  # every later electron's column of S
            elif what == "growth":
                C[t][:, o] *= 2.0 ** -6  # all of S: the ratios grow 64-fold
            elif t == 1:
                C[t][3, un[2]] = np.nan
    if what == "nan":
        md = W.double_well_paper(40)
        n, N, Ne = 3, 41, 20
        x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 5 * 9.5e-4, 1)
        occ = W.lowest_occupations(n, Ne)
        C = W.mixed_coefficients(occ, N, 2, 0.5)
        got = []
        for bad in (False, True):
            if bad:
                change(C, occ)
            ctx = P.Context(md, n, norm_tol=-1.0)
            ctx.set_state(x, p, occ, C)
            got.append(ctx.hop_probabilities(100.0))
            ctx.close()
        assert np.array_equal(got[0][[0, 2]], got[1][[0, 2]])
        assert np.all(got[1][1][:, Ne + 2] == 0.0)
        keep = [m for m in range(N) if m != Ne + 2]
        assert np.abs(got[0][1][:, keep] - got[1][1][:, keep]).max() <= 1e-12 * got[0][1].max()
        return
    _case(P, 50, 24, 0.5, change)
