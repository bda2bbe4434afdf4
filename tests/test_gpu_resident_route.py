"""GPU: solves go to the engine that is faster.  A range of few colours of an FP64 lattice that
runs on chip as a whole streams where the streamed pass is the faster one (its blocks have the
FP64 units to themselves), and larger ranges and FP32 ranges stay on chip; lattices at the line
where whole solves were measured slower on chip stream.  Ranges add up to the whole either way
(both engines stop at tol: 50 tol of the terms' magnitudes)."""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,dims,d,prec,few,many", [
    (L.LD_STENCIL_2D13_SQ, (300, 300), 2, L.LD_FP64, 1, 4),      # us an iteration: 3 colours 33 streamed, 59 on chip
    (L.LD_STENCIL_2D5, (300, 300), 4, L.LD_FP64, 1, 4),          # 30, 49
    (L.LD_STENCIL_3D7, (56, 56, 56), 2, L.LD_FP64, 1, 4),        # 50, 73
    (L.LD_STENCIL_2D13_SQ, (520, 520), 2, L.LD_MIXED, 4, 4),     # 25, 12
])
def test_ranges_take_the_faster_engine_and_add_up(kind, dims, d, prec, few, many):
    tol = 1e-8 if prec == L.LD_FP64 else 1e-6
    ctx = L.ld_create(L.grid_matrix(kind, dims, 0.3), d, 20, tol, L.options(precision=prec))
    whole, info = L.ld_logdet(ctx)
    terms, _ = L.ld_column_terms(ctx)
    nc = len(terms)
    assert info["engine"] == 4
    assert L.ld_logdet_partial(ctx, 2, 5)[1]["engine"] == few
    a, ia = L.ld_logdet_partial(ctx, 0, 3)
    b, ib = L.ld_logdet_partial(ctx, 3, nc)
    assert (ia["engine"], ib["engine"]) == (few, many)
    bar = 50 * tol if prec == L.LD_FP64 else 2e-5
    assert abs(a + b - whole) <= bar * np.abs(terms).sum()
    again, info = L.ld_logdet(ctx)                   # the same bits after the other engine's turn
    assert info["engine"] == 4 and again == whole


@pytest.mark.parametrize("kind,dims,d,prec,engine", [
    (L.LD_STENCIL_3D7, (60, 60, 60), 4, L.LD_MIXED, 1),          # 69 us streamed, 79 on chip
    (L.LD_STENCIL_3D7, (64, 64, 64), 4, L.LD_MIXED, 4),          # 79, 66
    (L.LD_STENCIL_3D7, (60, 60, 60), 6, L.LD_FP64, 1),           # 748, 806
    (L.LD_STENCIL_3D7, (64, 64, 64), 6, L.LD_FP64, 4),           # 1285, 1050
    (L.LD_STENCIL_2D13_SQ, (450, 443), 4, L.LD_MIXED, 1),        # 42, 45
    (L.LD_STENCIL_2D13_SQ, (520, 513), 2, L.LD_MIXED, 4),        # 29, 26
])
def test_whole_solves_at_the_line(kind, dims, d, prec, engine):
    ctx = L.ld_create(L.grid_matrix(kind, dims, 2.0), d, 12, 1e-4, L.options(precision=prec))
    assert L.ld_logdet(ctx)[1]["engine"] == engine
