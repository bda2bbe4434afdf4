"""GPU: calls that find no device memory for the resident engine's workspace take the streaming
route or report LD_ENOMEM, on the first call and on the ones after it, and use the resident
engine once there is memory again."""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def hold_all_but(free_bytes):
    """Device memory held until at most free_bytes are left (never touched)."""
    held = []
    for chunk in (1 << 30, 1 << 24, 1 << 21):
        while torch.cuda.mem_get_info()[0] - chunk >= free_bytes:
            k = (torch.cuda.mem_get_info()[0] - free_bytes) // chunk if chunk == 1 << 30 else 1
            held.append(torch.empty(int(k) * chunk, dtype=torch.uint8, device="cuda"))
    return held


def test_vector_form_without_room_for_its_records_streams_every_time():
    dims = (64, 64)
    V = synth.random_probe_block(3, int(np.prod(dims)), 1)
    make = lambda engine: L.ld_create(L.grid_matrix(L.LD_STENCIL_2D5, dims, 0.3), 1, 20, 1e-9, L.options(engine=engine))
    ref, _ = L.ld_logmv(make(1), V)              # both routes' kernels are loaded
    L.ld_logmv(make(0), V)
    ctx = make(0)                                # its workspace (64 MB of records) is not there yet
    torch.cuda.empty_cache()
    held = hold_all_but(48 << 20)
    try:
        for _ in range(3):
            Y, info = L.ld_logmv(ctx, V)
            assert info["engine"] != 4
            assert np.linalg.norm(Y - ref) <= 50e-9 * np.linalg.norm(ref)
    finally:
        del held
        torch.cuda.empty_cache()
    Y, info = L.ld_logmv(ctx, V)
    assert info["engine"] == 4 and np.linalg.norm(Y - ref) <= 50e-9 * np.linalg.norm(ref)
