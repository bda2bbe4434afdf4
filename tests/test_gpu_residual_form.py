"""GPU: the reported residual of an FP64 solve is that of the x it returns, on the matrix as given.

One colour on a torus: v = 1, so x is a constant after one iteration, Q x = kappa^2 x, and the
residual is 1 - kappa^2 x with x = seed projection / n.  The solve itself forms (4 or 6 + kappa^2)
and so returns an x off by up to 1e-9 of itself here; a residual kernel that rounds kappa^2 the same
way would report zero.  Difference form: two roundings, 2^-52 of 1; two further iterations of the
resident engine move x by its own rounding, 2^-52 of x: 4 x 2^-52 in all.
"""
from fractions import Fraction

import numpy as np
import pytest

import paper_1105_5256_gb300 as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [0, 1])
@pytest.mark.parametrize("dims,k2", [((64, 48), 1.2345e-6), ((45, 31), 7e-7), ((12, 10, 9), 3.3e-7)])
def test_reported_residual_of_a_constant_solution(dims, k2, engine):
    kind = L.LD_STENCIL_2D5 if len(dims) == 2 else L.LD_STENCIL_3D7
    n = int(np.prod(dims))
    ctx = L.ld_create(L.grid_matrix(kind, dims, k2, periodic=True), 1, 12, 1e-6,
                      L.options(engine=engine, keep_x0=1, colouring=np.zeros(n, np.int32)))
    _, info = L.ld_logdet(ctx)
    assert info["iters"] == 1 and info["engine"] == (1 if engine else 4)
    x = L.ld_column_terms(ctx)[1][0] / n
    want = abs(float(1 - Fraction(k2) * Fraction(x)))
    bar = 4 * 2.0 ** -52
    assert want > 1000 * bar                     # the two forms can be told apart
    assert abs(info["rel_resid_max"] - want) <= bar
