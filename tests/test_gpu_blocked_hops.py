"""Hop probabilities of the mixed path by blocked Gauss-Jordan elimination
(csrc/iesh_hop_bj.cu) against the oracle's determinant ratios, at the edges
of its blocks of four slots, column groups of eight, warps and its range."""
import numpy as np
import pytest

import iesh_inputs as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


# (M, Ne): one electron, a short last block, one and two electrons past a
# column group, all orbitals but one occupied, the largest size and the
# first size past it
@pytest.mark.parametrize("M,Ne", [(1, 1), (2, 2), (5, 4), (8, 7), (9, 9), (17, 8), (31, 16), (40, 33), (63, 31), (64, 33),
                                  (95, 47), (95, 48), (96, 48), (70, 1)])
def test_hop_probabilities(P, M, Ne):
    """FP32 ratios: 2e-6 of the largest probability, the mixed path's bound,
    scaled by the condition of the overlap matrix where it is above 10."""
    md = W.double_well_paper(40)
    md.update(M=M, Ne=Ne)
    n, dt, N = 5, 100.0, M + 1
    x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 5 * 9.5e-4, M)
    occ = W.random_occupations(n, N, Ne, M + 1)
    C = W.mixed_coefficients(occ, N, M + 2, 0.8)
    ctx = P.Context(md, n, precision=P.PREC_MIXED)
    ctx.set_state(x, p, occ, C.astype(np.complex64))
    g = ctx.hop_probabilities(dt)
    ctx.run(dt, 40, seed=3)
    st = ctx.get_state()
    ctx.close()
    assert np.all(st["status"] & 0x2 == 0)
    B = O.bind(md)
    for t in range(n):
        d = O.eigen(B, x[t])[3]
        ref = O.hop_probs(occ[t], C[t].T, d, p[t] / md["mass"], dt)[0]
        cond = np.linalg.cond(C[t].T[occ[t]])
        assert np.abs(g[t] - ref).max() <= 2e-6 * max(1.0, cond / 10) * max(np.abs(ref).max(), 1e-300)


def test_singular_and_certain(P):
    """A zero overlap row sets the singular bit and gives no probabilities; a
    huge probability (beyond 1) takes the first slot that reaches it, as the
    slot-by-slot sums do."""
    md = W.double_well_paper(40)
    n, N, Ne = 3, 41, 20
    x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 5 * 9.5e-4, 1)
    occ = W.lowest_occupations(n, Ne)
    C = W.mixed_coefficients(occ, N, 2, 0.8)
    C[0, :, 3] = 0.0  # orbital 3 is occupied: its row of S vanishes
    out = []
    for hop in (0, 256):
        ctx = P.Context(md, n, precision=P.PREC_MIXED, norm_tol=-1.0)
        ctx.set_kernel_shape(0, 0, hop)
        ctx.set_state(x, p * 1e5, occ, C.astype(np.complex64))
        out.append(ctx.hop_probabilities(100.0))
        ctx.close()
    assert np.all(out[0][0] == 0.0)
    assert out[0][1:].max() > 1.0
    for t in (1, 2):
        assert np.abs(out[0][t] - out[1][t]).max() <= 2e-6 * np.abs(out[1][t]).max() * 10
