"""Mixed-precision propagation on the tensor cores for 128 < N <= 256
(csrc/iesh_cheb_tcl.cu): one step against the oracle at the edges of its row
tiles, electron blocks and digit counts, its column scales, and the line to
the SIMT kernel."""
import numpy as np
import pytest

import iesh_inputs as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2212_00518_gb300 as pkg
    return pkg


def _state(md, n, seed, kT=0.0075):
    N = md["M"] + 1
    x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], kT, seed)
    occ = W.random_occupations(n, N, md["Ne"], seed + 1)
    return x, p, occ, W.mixed_coefficients(occ, N, seed + 2, 0.5)


def _one_step(P, md, x, p, occ, C, dt, shape=None):
    ctx = P.Context(md, x.shape[0], precision=P.PREC_MIXED)
    if shape:
        ctx.set_kernel_shape(*shape, 0)
    ctx.set_state(x, p, occ, C.astype(np.complex64))
    ctx.run(dt, 1, seed=5)
    st = ctx.get_state()
    st["K"] = ctx.propagator_terms()
    ctx.close()
    return st


def _tol(K):
    # K orders of unit-norm columns: each rounds four FP32 results (2^-24), and
    # the recurrence carries an order's error to the sum at most k-fold; the
    # coefficients, couplings and phases are rounded to FP32 once (a few 2^-24)
    return (2.0 * K * (K + 1) + 16) * 2.0 ** -24


# (M, Ne): N = 129 (one row in the second tile), 160 and 161 (a warp of rows
# more), 192 (the line for few electrons), 201, 255, 256; electrons: the
# fewest on the tensor cores and one fewer, one block and one more, the most
@pytest.mark.parametrize("M,Ne", [(128, 16), (128, 15), (128, 64), (159, 17), (160, 33), (190, 6), (191, 6), (191, 5),
                                  (200, 100), (254, 31), (255, 112), (255, 8)])
def test_one_step_against_oracle(P, M, Ne):
    md = W.double_well(M, Ne)
    n = 3
    x, p, occ, C = _state(md, n, M + Ne)
    st = _one_step(P, md, x, p, occ, C, 1.0)
    assert np.all(st["status"] == 0)
    B = O.bind(md)
    for t in range(n):
        r = O.step_one(B, x[t], p[t], occ[t].astype(np.int32), C[t].T, 1.0, seed=5, traj=t, n=0)
        assert np.abs(st["C"][t].T - r["C"]).max() <= _tol(st["K"][t])


# couplings from none to strong: one to three digits, W' resident and streamed
@pytest.mark.parametrize("M", [128, 200, 255])
@pytest.mark.parametrize("kick,Gamma", [(1.0, 0.0), (1.0, 1e-3), (50.0, 0.05), (500.0, 0.5)])
def test_coupling_range_against_oracle(P, M, kick, Gamma):
    md = W.double_well(M, 20)
    md["Gamma"] = Gamma
    n = 2
    x, p, occ, C = _state(md, n, 7)
    st = _one_step(P, md, x, p * kick, occ, C, 1.0)
    B = O.bind(md)
    for t in range(n):
        r = O.step_one(B, x[t], p[t] * kick, occ[t].astype(np.int32), C[t].T, 1.0, seed=5, traj=t, n=0)
        assert np.abs(st["C"][t].T - r["C"]).max() <= _tol(st["K"][t])


@pytest.mark.parametrize("shape", [None, (4, 1), (4, 3)])
def test_column_scales(P, shape):
    """Columns scaled by powers of two give exactly scaled results, a NaN stays
    in its column, and the blocks' width (a requested shape) does not matter."""
    md = W.double_well(140, 20)
    x, p, occ, C = _state(md, 2, 3)
    C = C.astype(np.complex64).astype(np.complex128)
    ref = _one_step(P, md, x, p, occ, C, 1.0)["C"]
    k = np.arange(20) % 7 * 9 - 27
    scaled = C * np.ldexp(1.0, k)[None, :, None]
    scaled[1, 5, 50] = np.nan
    got = _one_step(P, md, x, p, occ, scaled, 1.0, shape)["C"]
    assert np.isnan(got[1, 5]).all()
    back = got * np.ldexp(1.0, -k)[None, :, None]
    assert np.array_equal(back[0], ref[0])
    assert np.array_equal(np.delete(back[1], 5, 0), np.delete(ref[1], 5, 0))


def test_range_of_trajectories_is_bit_identical(P):
    """A trajectory's electrons go to several CTAs in a small batch and to one
    in a large batch: the bits are the same."""
    md = W.double_well(140, 60)
    n = 330
    x, p, occ, C = _state(md, n, 11)
    full = _one_step(P, md, x, p, occ, C, 1.0)["C"]
    few = _one_step(P, md, x[:3], p[:3], occ[:3], C[:3], 1.0)["C"]
    assert np.array_equal(full[:3], few)
