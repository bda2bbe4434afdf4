"""GPU: the resident engines' device waits end.  A record nobody writes and a barrier phase
nobody completes run into their limit; a team one of whose CTAs is left out of the launch gives
up and the call returns LD_ETIMEOUT; the context then solves as before, to the bit."""
import time

import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu


def gives_up(ctx, limit_ns=30_000_000):
    t0 = time.perf_counter()
    with pytest.raises(L.LogDetError) as e:
        L.ld_team_wait_selftest(ctx, limit_ns)
    assert e.value.status == L.LD_ETIMEOUT
    assert time.perf_counter() - t0 < 2.0


def test_every_kind_of_wait_is_bounded():
    with pytest.raises(L.LogDetError) as e:
        L.ld_wait_selftest(20_000_000)
    assert e.value.status == L.LD_ETIMEOUT
    assert "bulk copy, record, cluster barrier" in str(e.value)


@pytest.mark.parametrize("keep", [0, 1])
def test_a_lattice_team_without_its_last_cta_gives_up(keep):
    ctx = L.ld_create(L.grid_matrix(L.LD_STENCIL_2D13_SQ, (200, 150), 0.3), 2, 20, 1e-8, L.options(keep_x0=keep))
    v, info = L.ld_logdet(ctx)
    assert info["engine"] == 4
    gives_up(ctx)
    assert L.ld_logdet(ctx)[0] == v


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
def test_a_csr_team_without_its_last_cta_gives_up(prec):
    n = 3001
    rp, ci, vv = synth.csr_from_edges(n, *synth.random_sparse_spd_pattern(9, n), 0.3)
    ctx = L.ld_create(L.csr_matrix(rp, ci, vv), 1, 16, 1e-6, L.options(precision=prec))
    v, info = L.ld_logdet(ctx)
    assert info["engine"] == 4
    gives_up(ctx)
    assert L.ld_logdet(ctx)[0] == v


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
def test_a_csr_team_gives_up_with_empty_colour_classes(prec):
    """A caller's colouring with gaps: of the first 200 colours the odd ones are empty, the others
    have a vertex each.  A team solves at most 152 colours at a time over a launch, in tiles of an
    even number, so odd owners start with an empty class and have vectors in later rounds."""
    n = 640
    rp, ci, vv = synth.csr_from_edges(n, *synth.random_sparse_spd_pattern(9, n), 0.3)
    col = np.concatenate([np.arange(0, 200, 2), np.arange(200, 740)]).astype(np.int32)
    ctx = L.ld_create(L.csr_matrix(rp, ci, vv), 1, 16, 1e-6, L.options(precision=prec, colouring=col))
    v, info = L.ld_logdet(ctx)
    assert info["engine"] == 4 and info["n_colours"] == 740
    gives_up(ctx)
    assert L.ld_logdet(ctx)[0] == v


@pytest.mark.parametrize("keep", [0, 1])
@pytest.mark.parametrize("csr", [False, True])
def test_a_solve_whose_teams_gave_up_goes_on_on_the_other_engine(csr, keep):
    """As ld_logdet does when a team's CTAs become resident piecemeal: the value and seed
    solutions of the one-CTA engine (both stop at tol: 50 tol of the terms' magnitudes)."""
    if csr:
        rp, ci, vv = synth.csr_from_edges(3001, *synth.random_sparse_spd_pattern(9, 3001), 0.3)
        make = lambda engine: L.ld_create(L.csr_matrix(rp, ci, vv), 1, 16, 1e-8, L.options(engine=engine, keep_x0=keep))
    else:
        make = lambda engine: L.ld_create(L.grid_matrix(L.LD_STENCIL_2D13_SQ, (200, 150), 0.3), 2, 20, 1e-8,
                                          L.options(engine=engine, keep_x0=keep))
    ctx, ref = make(0), make(2)
    want, _ = L.ld_logdet(ref)
    terms, _ = L.ld_column_terms(ref)
    first, info = L.ld_logdet(ctx)
    assert info["engine"] == 4
    got, info = L.ld_team_wait_selftest(ctx, 30_000_000, go_on=True)
    assert info["engine"] == 2 and abs(got - want) <= 50e-8 * np.abs(terms).sum()
    if keep:
        assert np.allclose(L.ld_grad(ctx, [L.LD_P_SCALE]), L.ld_grad(ref, [L.LD_P_SCALE]), rtol=50e-8, atol=0)
    again, info = L.ld_logdet(ctx)
    assert info["engine"] == 4 and again == first


def test_the_self_test_needs_teams():
    ctx = L.ld_create(L.grid_matrix(L.LD_STENCIL_2D5, (32, 16), 0.5), 1, 16, 1e-8, L.options(engine=1))
    with pytest.raises(L.LogDetError) as e:
        L.ld_team_wait_selftest(ctx, 30_000_000)
    assert e.value.status == L.LD_EUNSUPPORTED
