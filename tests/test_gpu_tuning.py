"""The autotuner and the tensor-core propagators: their built-in shape is what it
compares with, and what it keeps where shapes can only narrow it."""
import numpy as np
import pytest

import iesh_inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,Ne,precision", [(27, 14, 0), (100, 50, 0), (200, 100, 0), (140, 20, 1), (20, 10, 0)])
def test_built_in_shape(M, Ne, precision):
    import paper_2212_00518_gb300 as P
    from paper_2212_00518_gb300 import tuning
    md = W.double_well(M, Ne)
    n = 16
    x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 0.0075, 1)
    occ = W.lowest_occupations(n, Ne)
    ctx = P.Context(md, n, precision=precision)
    C = W.mixed_coefficients(occ, M + 1, 2, 0.3).astype(ctx.cdtype)
    tensor_cores = M >= 27
    assert (ctx.kernel_shape()[0] == 0) == (tensor_cores and precision == 0)
    best = tuning.autotune(ctx, x, p, occ, C, 1.0, steps=1)
    timed = set(best["times"]["cheb"])
    ctx.close()
    if tensor_cores:
        assert "(0, 0)" in timed
    if tensor_cores and precision == 0:
        assert timed == {"(0, 0)"} and best["cheb"] == (0, 0)
