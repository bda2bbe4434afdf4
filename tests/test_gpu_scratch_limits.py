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
    for left in (free_bytes + (256 << 20), free_bytes):      # the second piece is large enough not to be rounded up
        size = (torch.cuda.mem_get_info()[0] - left) >> 21 << 21
        held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
    assert torch.cuda.mem_get_info()[0] <= free_bytes + (4 << 20)
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


def test_a_solve_without_room_for_its_exchange_buffers_takes_the_other_engine():
    p, t = synth.perturbed_triangulation(6, 141, 97)
    from paper_1105_5256_gb300 import mesh
    rp, ci, vv = mesh.spde_csr(p, t, 0.3 * 140 * 96, 2, 1.0)
    lo, hi = L.ld_csr_bounds(rp, ci, vv)
    make = lambda engine: L.ld_create(L.csr_matrix(rp, ci, vv), 2, 16, 1e-6,
                                      L.options(engine=engine, lambda_min=lo, lambda_max=hi))
    ref, info = L.ld_logdet(make(2))
    assert info["engine"] == 2
    ctx = make(0)                                # w of every team's vectors: 7 MB, allocated by the first solve
    torch.cuda.empty_cache()
    held = hold_all_but(4 << 20)
    try:
        for _ in range(2):
            v, info = L.ld_logdet(ctx)
            assert info["engine"] == 2 and abs(v - ref) <= 50e-6 * abs(ref)
    finally:
        del held
        torch.cuda.empty_cache()
    v, info = L.ld_logdet(ctx)
    assert info["engine"] == 4 and abs(v - ref) <= 50e-6 * abs(ref)


def test_vector_form_that_overruns_its_records_streams_at_once_from_then_on():
    """Records for n / 3 iterations here (1500 columns of 240 vertices), fewer than the solve takes."""
    dims, ncols = (16, 15), 1500
    n = int(np.prod(dims))
    V = synth.random_probe_block(3, n, ncols)
    make = lambda engine, k2: L.ld_create(L.grid_matrix(L.LD_STENCIL_2D13_SQ, dims, k2), 1, 20, 1e-10, L.options(engine=engine))
    Y1, info1 = L.ld_logmv(make(1, 1e-4), V)
    assert info1["iters"] > n // 3
    ctx = make(0, 1e-4)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    Y, first = L.ld_logmv(ctx, V)
    assert first["engine"] != 4 and np.linalg.norm(Y - Y1) <= 50e-10 * np.linalg.norm(Y1)
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20          # the records took 115 MB
    Y, second = L.ld_logmv(ctx, V)
    assert second["gpu_launches"] == first["gpu_launches"] - 2     # no attempt on chip any more
    assert np.linalg.norm(Y - Y1) <= 50e-10 * np.linalg.norm(Y1)
    L.ld_set_params(ctx, 50.0, 0.0, 1.0)
    Y, info = L.ld_logmv(ctx, V)
    W, _ = L.ld_logmv(make(1, 50.0), V)
    assert info["engine"] == 4 and np.linalg.norm(Y - W) <= 50e-10 * np.linalg.norm(W)
