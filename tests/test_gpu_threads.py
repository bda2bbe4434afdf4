"""GPU: contexts driven from threads of their own at once, over every form of the resident engine
(clusters, cooperative lattice and CSR teams, which take turns, the vector form, a batch) and the
streaming engine beside them, give the bits of the same calls one by one."""
import threading

import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu


def jobs():
    rp, ci, vv = synth.csr_from_edges(3001, *synth.random_sparse_spd_pattern(9, 3001), 0.3)
    V = synth.random_probe_block(2, 200 * 150, 2)
    grid = lambda kind, dims, k2, d, **kw: L.ld_create(L.grid_matrix(kind, dims, k2), d, 20, 1e-8, L.options(**kw))
    solve = lambda ctx: lambda: np.append(L.ld_column_terms(ctx)[0], L.ld_logdet(ctx)[0]) if L.ld_logdet(ctx) else None
    out = [solve(grid(L.LD_STENCIL_2D5, (61, 50), 0.3, 2)),                          # clusters
           solve(grid(L.LD_STENCIL_2D13_SQ, (200, 150), 0.3, 2)),                    # cooperative
           solve(grid(L.LD_STENCIL_2D13_SQ, (180, 170), 0.2, 2, keep_x0=1)),         # cooperative, with x
           solve(L.ld_create(L.csr_matrix(rp, ci, vv), 1, 16, 1e-8, L.options())),   # CSR teams
           solve(grid(L.LD_STENCIL_2D5, (150, 140), 0.3, 2, engine=1))]              # streamed
    ctx = grid(L.LD_STENCIL_2D13_SQ, (200, 150), 0.3, 1)
    out.append(lambda: L.ld_invsqrt_mv(ctx, V)[0])
    b = L.ld_batch_create([L.grid_matrix(L.LD_STENCIL_2D5, (s, s), 0.2) for s in (40, 90, 150)], [2, 2, 2], 20, 1e-8, L.options())
    out.append(lambda: L.ld_batch_logdet(b)[0])
    return out


def test_concurrent_contexts_give_the_serial_bits():
    calls = jobs()
    want = [np.array(f(), copy=True) for f in calls]
    errors = []

    def work(k):
        try:
            for _ in range(8):
                got = calls[k]()
                if not np.array_equal(got, want[k]):
                    errors.append((k, np.abs(got - want[k]).max()))
        except Exception as e:                       # reported by the main thread
            errors.append((k, repr(e)))
    pool = [threading.Thread(target=work, args=(k,)) for k in range(len(calls))]
    for t in pool:
        t.start()
    for t in pool:
        t.join()
    assert not errors, errors
