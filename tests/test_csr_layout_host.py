"""The host part of the CSR resident engine's layout (no GPU): what it costs to find that a matrix
is too large, and that a matrix that fits is laid out."""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth


def torus(nx, ny):
    return synth.csr_from_edges(nx * ny, *synth.torus_edges(nx, ny), 0.5)[:2]


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
def test_a_matrix_too_large_by_its_rows_alone_is_not_scanned(prec):
    # 152 CTAs of 4700 rows: at 54 bytes a row (four FP32 vectors) or 74 (two FP64) beyond 227 KB
    rp, ci = torus(900, 800)
    fits, _, scanned = L.ld_csr_layout(rp, ci, prec, 30, 20, 152)
    assert not fits and scanned == 0


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
def test_a_matrix_that_fits_is_laid_out(prec):
    rp, ci = torus(64, 64)
    fits, ctas, scanned = L.ld_csr_layout(rp, ci, prec, 25, 20, 152)
    assert fits and 1 < ctas <= 152 and 0 < scanned
