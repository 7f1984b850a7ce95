"""The hop that the mixed path's blocked kernel (csrc/iesh_hop_bj.cu) selects
and takes: against the LU kernel from the same coefficients and uniforms, over
totals from a few percent to far beyond 1, and the singular case."""
import numpy as np
import pytest

import iesh_inputs as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


def _step(P, md, x, p, occ, C, hop):
    ctx = P.Context(md, x.shape[0], precision=P.PREC_MIXED, norm_tol=-1.0)
    ctx.set_kernel_shape(0, 0, hop)
    ctx.set_state(x, p, occ, C)
    ctx.run(100.0, 1, seed=9)
    st = ctx.get_state()
    st["hops"], st["frus"] = ctx.counters()[1:]
    ctx.close()
    return st


# a short last block of slots, one and several column groups, the largest size
@pytest.mark.parametrize("M,Ne", [(5, 4), (17, 8), (40, 20), (95, 48)])
def test_selected_hops(P, M, Ne):
    md = W.double_well_paper(40)
    md.update(M=M, Ne=Ne)
    n, N = 3000, M + 1
    x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 5 * 9.5e-4, M)
    p = p * 10.0 ** (0.5 + 1.5 * (np.arange(n) % 16) / 15)
    occ = W.random_occupations(n, N, Ne, M + 1)
    C = W.mixed_coefficients(occ, N, M + 2, 0.8).astype(np.complex64)
    a, b = (_step(P, md, x, p, occ, C, hop) for hop in (0, 256))
    assert np.array_equal(a["C"], b["C"])
    assert np.all((a["status"] | b["status"]) & P.iesh.TRAJ_SINGULAR == 0)
    # the two kernels' probabilities differ by about 10^-6 of the total, and a
    # hop differs where the uniform falls between two such running sums: 0.003
    # of 3000 expected, three or more are not seen
    same = (a["occ"] == b["occ"]).all(1) & (a["hops"] == b["hops"]) & (a["frus"] == b["frus"])
    assert np.count_nonzero(~same) <= 2
    # every slot has hopped, the last among them, and the outermost orbitals
    # have been reached
    slots, reached = set(), set()
    for t in np.flatnonzero(b["hops"] == 1):
        old, new = set(occ[t]), set(b["occ"][t])
        slots.add(int(np.searchsorted(np.sort(occ[t]), (old - new).pop())))
        reached.add(int((new - old).pop()))
    assert slots == set(range(Ne)) and {0, N - 1} <= reached


def test_singular_overlap_takes_no_hop(P):
    """An electron without amplitude: the singular bit after a step, no hop,
    and the neighbours as without it."""
    md = W.double_well_paper(40)
    n, N, Ne = 4, 41, 20
    x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 5 * 9.5e-4, 1)
    occ = W.random_occupations(n, N, Ne, 2)
    C = W.mixed_coefficients(occ, N, 3, 0.8).astype(np.complex64)
    ref = _step(P, md, x, p * 30, occ, C, 0)
    C[1, 7] = 0.0
    for hop in (0, 256):
        st = _step(P, md, x, p * 30, occ, C, hop)
        assert st["status"][1] & P.iesh.TRAJ_SINGULAR
        assert st["hops"][1] == 0 and np.array_equal(st["occ"][1], np.sort(occ[1]))
        if hop == 0:
            for t in (0, 2, 3):
                assert np.array_equal(st["occ"][t], ref["occ"][t]) and st["status"][t] == ref["status"][t]
