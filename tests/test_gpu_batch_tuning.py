"""GPU: a batch's tile width is tuned on the instances that will use it.  Beside many instances of
the resident engine, one lattice too wide for any cluster (lines of 2100 vertices) must not put all
of them through trial contexts of the other engine: creating the batch costs at most what the two
parts cost by themselves, and half of that again."""
import time

import numpy as np
import pytest

import paper_1105_5256_gb300 as L

pytestmark = pytest.mark.gpu


def created(shapes, tol=1e-6):
    mats = [L.grid_matrix(L.LD_STENCIL_2D5, s, 0.05) for s in shapes]
    t = time.perf_counter()
    b = L.ld_batch_create(mats, [4] * len(shapes), 20, tol, L.options(precision=L.LD_MIXED))
    return time.perf_counter() - t, b


def test_creation_tunes_the_instances_that_need_a_width_alone():
    fits = lambda side: [(side + k, side) for k in range(40)]
    created(fits(64) + [(2100, 5)])                    # kernels loaded
    one, _ = created([(2100, 7)])
    many, _ = created(fits(300))
    both, b = created(fits(301) + [(2100, 9)])
    assert both <= 1.5 * (one + many), (one, many, both)
    vals, _, info = L.ld_batch_logdet(b)
    assert np.all(np.isfinite(vals)) and info["engine"] == 2
