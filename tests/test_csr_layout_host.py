"""The host part of the CSR resident engine's layout (no GPU): what it costs to find that a matrix
is too large, and that a matrix that fits is laid out."""
import os
import resource
import subprocess
import sys

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


def test_a_broken_pattern_is_refused():
    rp, ci = torus(8, 8)
    for r, c in ((rp + 1, ci), (rp[::-1].copy(), ci), (rp, np.where(np.arange(ci.size) == 7, 64, ci)), (rp, ci - 1)):
        with pytest.raises(L.LogDetError) as e:
            L.ld_csr_layout(r, c, L.LD_FP64, 4, 20, 152)
        assert e.value.status == L.LD_EINVAL


CHILD = """
import resource, sys
sys.path.insert(0, %r)
import paper_1105_5256_gb300 as L
from tests.test_csr_layout_host import torus
rp, ci = torus(250, 250)
want = L.ld_csr_layout(rp, ci, L.LD_MIXED, 30, 20, 152)
size = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (size + (64 << 20), resource.RLIM_INFINITY))
assert L.ld_csr_layout(rp, ci, L.LD_MIXED, 30, 20, 152) == want and want[0]
print("ok")
"""


def test_a_process_that_can_start_no_thread_lays_out_on_its_own():
    """The layout of a larger matrix uses threads; where none can be started (here their 256 MB stacks
    exceed the address space that is left) the calling thread does it, and nothing is thrown."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    hard = resource.getrlimit(resource.RLIMIT_STACK)[1]
    big = 256 << 20
    if hard != resource.RLIM_INFINITY and hard < big:
        pytest.skip("the stack limit cannot be raised")
    r = subprocess.run([sys.executable, "-c", CHILD % root], capture_output=True, text=True, timeout=300, cwd=root,
                       env=dict(os.environ, OPENBLAS_NUM_THREADS="1"),
                       preexec_fn=lambda: resource.setrlimit(resource.RLIMIT_STACK, (big, hard)))
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr[-2000:]
