"""GPU parity of the true-residual sweep of the 5- and 7-point lattices (reliable updates and
the reported residual) at the edges of its warps, blocks and segments.

The same matrix as a CSR context takes the general residual kernel.  Both solves stop at
tol 1e-2, so the reported max_k ||v_k - Q x_k|| / ||v_k|| is far above rounding: in FP64 the
two iterates agree to ~1e-11 and the residuals to 1e-8 of themselves; FP32 vectors move x by
~1e-7 |x|, which through |Q||x| <~ 60 moves the residual by ~1e-5 against 1e-2..1e-3.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu


def lattice_csr(dims, per, diag, scale):
    n = int(np.prod(dims))
    Q = sp.diags(diag).tocsr()
    stride = 1
    for d in dims:                                       # first axis fastest
        ring = sp.lil_matrix((d, d))
        for i in range(d):
            ring[i, i] += 2.0
            for j in (i - 1, i + 1):
                if per or 0 <= j < d:
                    ring[i, j % d] -= 1.0
        Q = Q + sp.kron(sp.kron(sp.eye(n // (stride * d)), ring), sp.eye(stride))
        stride *= d
    Q = sp.csr_matrix(Q)                                 # the context applies the scale
    Q.sort_indices()
    return L.csr_matrix(Q.indptr, Q.indices, Q.data, scale=scale)


@pytest.mark.parametrize("prec,delta,T,rtol", [
    (L.LD_FP64, 0.0, 2, 1e-8), (L.LD_FP64, 0.5, 4, 1e-8), (L.LD_MIXED, 0.0, 6, 1e-2), (L.LD_MIXED, 0.5, 2, 1e-2)])
@pytest.mark.parametrize("dims,per", [
    ((1, 5), False), ((3, 3), True), ((31, 9), True), ((33, 17), False), ((256, 40), True), ((257, 33), False),
    ((300, 70), False), ((9, 8, 7), True), ((33, 9, 5), False), ((64, 17, 3), True), ((5, 1, 6), False),
    ((40, 24, 18), False)])
def test_reported_residual_matches_the_general_kernel(dims, per, prec, delta, T, rtol):
    kind = L.LD_STENCIL_2D5 if len(dims) == 2 else L.LD_STENCIL_3D7
    n, k2, tau, scale = int(np.prod(dims)), 0.02, 0.5, 1.3
    mask = synth.obs_mask(4, n, 0.3)
    col, _ = L.ld_colour_grid(kind, dims, per, 2)

    def resid(matrix):
        ctx = L.ld_create(matrix, 2, 12, 1e-2, L.options(
            precision=prec, engine=1, tile_width=T, colouring=col, reliable_delta=delta, chunk_iters=4, keep_x0=1,
            lambda_min=scale * k2, lambda_max=scale * (4 * len(dims) + k2 + tau)))
        return L.ld_logdet(ctx)[1]["rel_resid_max"]
    got = resid(L.grid_matrix(kind, dims, k2, periodic=per, tau=tau, obs_mask=mask, scale=scale))
    want = resid(lattice_csr(dims, per, k2 + tau * np.asarray(mask, float), scale))
    assert want > 0
    if n > 200:                                          # tiny grids solve exactly: only rounding is left
        assert abs(got - want) <= rtol * want
    else:
        assert abs(got - want) <= rtol * want + (1e-13 if prec == L.LD_FP64 else 1e-6)
