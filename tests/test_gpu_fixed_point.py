"""FP64 propagation on the tensor cores in fixed point (csrc/iesh_cheb_fx.cu):
one step against the oracle at the edges of its row tiles, column blocks and
digit counts, and its column scales."""
import numpy as np
import pytest

import iesh_inputs as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu

# Tolerance of one step: K Chebyshev orders of unit-norm columns, each adding
# a few 2^-56, and the oracle's own Jacobi eigensolver, O(N) rotations per
# entry of 2^-53 each: below 256 x 16 x 2^-53 = 5e-13 in total.
TOL = 5e-13


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
    ctx = P.Context(md, x.shape[0])
    if shape:
        ctx.set_kernel_shape(*shape, 0)
    ctx.set_state(x, p, occ, C)
    ctx.run(dt, 1, seed=5)
    st = ctx.get_state()
    ctx.close()
    return st


# (M, Ne): N = 28 (the smallest), 32 and 33, 64 and 65, 128 and 129 (one and
# two row tiles), 256; one electron more than a column block holds; the
# largest Ne; fewest electrons on the tensor cores at N = 128
@pytest.mark.parametrize("M,Ne", [(27, 14), (31, 15), (32, 31), (63, 32), (64, 33), (100, 50), (127, 4), (127, 65),
                                  (128, 64), (199, 17), (255, 112)])
def test_one_step_against_oracle(P, M, Ne):
    md = W.double_well(M, Ne)
    n = 3
    x, p, occ, C = _state(md, n, M + Ne)
    st = _one_step(P, md, x, p, occ, C, 1.0)
    assert np.all(st["status"] == 0)
    B = O.bind(md)
    for t in range(n):
        r = O.step_one(B, x[t], p[t], occ[t].astype(np.int32), C[t].T, 1.0, seed=5, traj=t, n=0)
        assert np.abs(st["C"][t].T - r["C"]).max() <= TOL


# couplings from none to strong (the number of digits), long steps (many
# orders): paper model with dt = 100, double well at Gamma = 0
@pytest.mark.parametrize("case", ["none", "weak", "strong", "long"])
def test_coupling_range_against_oracle(P, case):
    if case == "long":
        md, dt = W.double_well_paper(140), 100.0
    else:
        md, dt = W.double_well(60), 1.0
        md["Gamma"] = {"none": 0.0, "weak": 1e-9, "strong": 0.5}[case]
        md["par"] = [0.002, 20.6 if case != "strong" else 2.0, -0.0038]
    n = 3
    x, p, occ, C = _state(md, n, 7)
    if case == "strong":
        p = p * 50
    st = _one_step(P, md, x, p, occ, C, dt)
    B = O.bind(md)
    for t in range(n):
        r = O.step_one(B, x[t], p[t], occ[t].astype(np.int32), C[t].T, dt, seed=5, traj=t, n=0)
        # the norm-wise bound, relative to the interval's length in orders
        assert np.abs(st["C"][t].T - r["C"]).max() <= TOL * max(1.0, dt / 10)


@pytest.mark.parametrize("shape", [None, (1, 1), (2, 4)])
def test_column_scales(P, shape):
    """Each electron's column has its own power-of-two scale: columns scaled
    by powers of two give exactly scaled results (also far outside the FP32
    range, up to the coarser scale taken there), a NaN stays in its column,
    and the blocks' width (a requested shape) does not matter."""
    md = W.double_well(100, 20)
    x, p, occ, C = _state(md, 2, 3)
    ref = _one_step(P, md, x, p, occ, C, 1.0)["C"]
    k = np.arange(20) % 7 * 9 - 27
    k[0], k[1] = 400, -400
    scaled = C * np.ldexp(1.0, k)[None, :, None]
    scaled[1, 5, 50] = np.nan
    got = _one_step(P, md, x, p, occ, scaled, 1.0, shape)["C"]
    assert np.isnan(got[1, 5]).all()
    assert np.isfinite(got[0]).all() and np.isfinite(np.delete(got[1], 5, 0)).all()
    back = got * np.ldexp(1.0, -k)[None, :, None]
    assert np.array_equal(back[0, 2:], ref[0, 2:])
    assert np.abs(back[0, :2] - ref[0, :2]).max() <= TOL


def test_range_of_trajectories_is_bit_identical(P):
    """The column blocks of a trajectory go to several CTAs in a small batch
    and to one in a large batch: the bits are the same."""
    md = W.double_well(128, 60)
    n = 160
    x, p, occ, C = _state(md, n, 11)
    full = _one_step(P, md, x, p, occ, C, 1.0)["C"]
    few = _one_step(P, md, x[:3], p[:3], occ[:3], C[:3], 1.0)["C"]
    assert np.array_equal(full[:3], few)
