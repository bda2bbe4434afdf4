"""GPU: the replay of the vector form hands alpha and beta of one iteration at a time to every
warp of a clustered team.  A warp that took the next iteration's would change its part of
log(Q) V, so many columns over one-CTA and several-CTA clusters, with more work in some CTAs
than in others, give the same bits on every call and the value of the shifted directions
(both stop each shift at a relative residual tol: 50 tol; FP32 vectors 2e-5).
"""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
@pytest.mark.parametrize("points,dims,per,ncols", [
    (L.LD_STENCIL_2D5, (16, 5), False, 200),         # one CTA, no boundary rows to wait for
    (L.LD_STENCIL_2D13_SQ, (40, 11), False, 170),
    (L.LD_STENCIL_2D5, (64, 61), True, 160),
    (L.LD_STENCIL_2D13_SQ, (100, 67), False, 40),    # blocks of uneven height
    (L.LD_STENCIL_3D7, (17, 13, 11), False, 60),
])
def test_replay_gives_the_same_bits_and_the_right_value(points, dims, per, ncols, prec):
    tol = 1e-9 if prec == L.LD_FP64 else 1e-6
    V = synth.random_probe_block(5, int(np.prod(dims)), ncols)
    make = lambda engine: L.ld_create(L.grid_matrix(points, dims, 0.3, periodic=per), 1, 20, tol,
                                      L.options(precision=prec, engine=engine))
    ctx = make(0)
    Y, info = L.ld_logmv(ctx, V)
    assert info["engine"] == 4
    for _ in range(10):
        assert np.array_equal(L.ld_logmv(ctx, V)[0], Y)
    W = L.ld_logmv(make(1), V)[0]
    bar = 50 * tol if prec == L.LD_FP64 else 2e-5
    assert np.all(np.linalg.norm(Y - W, axis=0) <= bar * np.linalg.norm(W, axis=0))
