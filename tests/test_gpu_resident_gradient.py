"""GPU: exactness of the FP32 Matern gradient on the resident engine.

The gradient sums x = Q^{-1} v over the probing vectors.  The roundings of x += alpha p and a
w that drifts from Q p both reach it; with compensated x and w formed from p what is left is
the residual's own rounding, below a few FP32 units (eps = 6e-8) of the gradient: 8 eps here,
against the FP64 solve of the same vectors (its own error, tol 1e-10, is far below).
"""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,per", [((150, 120), False), ((61, 83), False), ((64, 48), True), ((290, 210), False)])
def test_fp32_matern_gradient(dims, per):
    col, _ = L.ld_colour_grid(L.LD_STENCIL_2D13_SQ, dims, per, 2)
    err = []
    for k2 in (0.1, 0.105, 0.11):
        def grad(prec, tol):
            ctx = L.ld_create(L.grid_matrix(L.LD_STENCIL_2D13_SQ, dims, k2, periodic=per), 2, 20, tol,
                              L.options(precision=prec, colouring=col))
            _, g, info = L.ld_logdet_grad(ctx, [L.LD_P_KAPPA2, L.LD_P_SCALE])
            return np.asarray(g), info
        g32, info = grad(L.LD_MIXED, 1e-6)
        g64, _ = grad(L.LD_FP64, 1e-10)
        assert info["engine"] == 4
        err.append(np.linalg.norm(g32 - g64) / np.linalg.norm(g64))
    assert max(err) <= 8 * 6e-8
