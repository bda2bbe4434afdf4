"""GPU: the CSR resident engine's sums over lanes, warps and CTAs lose no bits to FP32.

A diagonal matrix of FP32 numbers 1 + k 2^-23 with one colour: v^T v = n and v^T Q v = sum of the
diagonal, a row a thread, so that nothing is rounded before the sums over threads.  At tol 0.9 the
solve ends after one iteration with the seed projection alpha n = n^2 / sum.  FP32 sums over a
warp's lanes would leave 1e-8; sums that carry their errors 2^-46 a step, 1e-12 with room.
"""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
@pytest.mark.parametrize("n", [33, 700, 20011, 40000])
def test_first_step_length_is_exact(n, prec):
    d = 1.0 + synth.rng(n).integers(0, 1 << 23, n) * 2.0 ** -23
    ctx = L.ld_create(L.csr_matrix(np.arange(n + 1), np.arange(n), d), 1, 12, 0.9,
                      L.options(precision=prec, colouring=np.zeros(n, np.int32), lambda_min=1.0, lambda_max=2.0))
    _, info = L.ld_logdet(ctx)
    assert info["engine"] == 4 and info["iters"] == 1
    seed = L.ld_column_terms(ctx)[1][0]
    assert abs(seed - n * (n / d.sum())) <= 1e-12 * n


@pytest.mark.parametrize("engine", [0, 1])
def test_dots_beyond_fp32_are_reported(engine):
    """|w|^2 of entries 1e20 overflows FP32: infinite, and so is the predicted residual."""
    n = 700
    d = 1e20 * (1.0 + synth.rng(n).random(n))
    ctx = L.ld_create(L.csr_matrix(np.arange(n + 1), np.arange(n), d), 1, 12, 0.5,
                      L.options(precision=L.LD_MIXED, engine=engine, colouring=np.zeros(n, np.int32), lambda_min=1e20, lambda_max=2e20))
    with pytest.raises(L.LogDetError) as e:
        L.ld_logdet(ctx)
    assert e.value.status == L.LD_ENUMERIC
