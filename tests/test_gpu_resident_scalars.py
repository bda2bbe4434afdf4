"""GPU: alpha and beta of the resident engines against the host's correctly rounded quotients.

The engine's quotient is off by at most 2^-51 of a unit in the last place before its last
rounding, so over random operands the chance of any difference from the correctly rounded one
is below 1e-9; outside [2^-400, 2^400] it calls the division, where nothing may differ.  beta is
compared as the quotient of the rho that was returned.  For FP32 vectors the quotients are left
1.5 units in the last place, and one rounding, off."""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu


def draw(seed, count, lo, hi):
    g = synth.rng(seed)
    return np.ldexp(1.0 + g.random(count), g.integers(lo, hi + 1, count))


@pytest.mark.parametrize("lo,hi", [(0, 0), (-30, 30), (-399, 398), (-404, -396), (396, 404), (-1000, 1000)])
def test_quotients_are_correctly_rounded(lo, hi):
    m = 200_000
    rr, pw = draw(1, m, lo, hi), draw(2, m, lo, hi)
    with np.errstate(over="ignore", under="ignore", invalid="ignore", divide="ignore"):
        # r.w and |w|^2 of a residual that falls by a random factor: rho = rr (1 - 2 a + a^2 b)
        rw = pw * synth.rng(3).uniform(0.1, 0.6, m)
        ww = rw * (rw / rr)
        out = L.ld_scalar_selftest(np.stack([rr, pw, rw, ww], 1))
        alpha, beta, rho = out[:, 0], out[:, 1], out[:, 2]
        fine = np.isfinite(rw) & np.isfinite(ww)
        assert fine.sum() > m // 4 and not out[fine, 3].any()
        assert np.array_equal(alpha, rr / pw)
        # the corrected quotient needs a residual above the subnormals; rho that small is only reached by cancellation
        ok = fine & np.isfinite(rho) & ((rho == 0) | (rho > 1e-280))
        assert np.array_equal(beta[ok], (rho / rr)[ok])
        size = np.abs(rr) + np.abs(2 * alpha * rw) + alpha * alpha * ww
        want = rr + alpha * (alpha * ww - 2.0 * rw)
        see = fine & np.isfinite(size) & (alpha * ww > 1e-280)
        assert np.all(np.abs(rho - np.maximum(want, 0.0))[see] <= 8 * 2.0 ** -53 * size[see])


@pytest.mark.parametrize("lo,hi", [(0, 0), (-399, 398), (-1000, 1000)])
def test_quotients_for_fp32_vectors(lo, hi):
    """Without the corrections: alpha within 2 units (1.5 and its last rounding), beta as the quotient
    of the rho it was formed from, itself formed from that alpha."""
    m = 100_000
    rr, pw = draw(4, m, lo, hi), draw(5, m, lo, hi)
    with np.errstate(over="ignore", under="ignore", invalid="ignore", divide="ignore"):
        rw = pw * synth.rng(6).uniform(0.1, 0.6, m)
        ww = rw * (rw / rr)
        out = L.ld_scalar_selftest(np.stack([rr, pw, rw, ww], 1), L.LD_MIXED)
        q = rr / pw
        normal = (q > 1e-300) & (q < 1e300)
        assert np.all(np.abs(out[:, 0] - q)[normal] <= 2 * 2.0 ** -52 * q[normal])
        ok = normal & np.isfinite(ww) & (out[:, 2] > 1e-280) & np.isfinite(out[:, 2] / rr)
        b = (out[:, 2] / rr)[ok]
        assert ok.sum() > m // 4 and np.all(np.abs(out[ok, 1] - b) <= 2 * 2.0 ** -52 * b)


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
def test_special_dots(prec):
    inf, nan, tiny = np.inf, np.nan, 5e-324
    rows = np.array([
        [1.0, 0.0, 0.0, 0.0], [1.0, -0.0, 1.0, 1.0], [1.0, -2.0, 1.0, 1.0],       # p.w not positive: not SPD
        [1.0, nan, 1.0, 1.0], [1.0, -inf, 1.0, 1.0],                              # not a number
        [0.0, 1.0, 0.0, 0.0],                                                     # converged exactly
        [tiny, 1.0, 0.0, 0.0], [1e-310, 1e-310, 0.5e-310, 0.3e-310],              # subnormal residual
        [1e300, 1e-300, 1.0, 1.0],                                                # alpha overflows
        [1.0, 3.0, 100.0, 1.0],                                                   # predicted norm below zero: 0
    ])
    out = L.ld_scalar_selftest(rows, prec)
    assert list(out[:, 3]) == [L.LD_ENOTSPD] * 3 + [L.LD_ENUMERIC] * 2 + [0] * 5
    assert not out[:5, :2].any()
    assert out[5, 0] == 0.0 and out[5, 1] == 0.0 and out[5, 2] == 0.0
    assert out[6, 0] == tiny and out[6, 1] == 1.0
    assert out[7, 0] == 1.0 and out[7, 1] == out[7, 2] / 1e-310 and 0.0 < out[7, 1] < 1.0
    assert np.isinf(out[8, 0])
    assert abs(out[9, 0] - 1.0 / 3.0) <= (1e-16 if prec == L.LD_MIXED else 0.0) and out[9, 1] == 0.0 and out[9, 2] == 0.0
