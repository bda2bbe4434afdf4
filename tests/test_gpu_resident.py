"""GPU parity of the resident engine (options.engine = 0 on grid kinds: a probing vector's
whole solve on chip, info engine 4) with the streaming grid engine on the same problem,
over geometries where its blocks, teams and exchanges can go wrong: lines that are no
multiple of 16 bytes, one line or one group a CTA, torus wraps onto the same CTA, teams of
one to sixteen CTAs in a cluster and cooperative teams over L2, blocks of a 3D lattice with
uneven sides, kappa^2 fields and masks, the kept seed solution, more shifts than lanes.

Both engines run the same recurrences to the same stopping rule (each shifted residual
<= tol), so terms and seed projections differ by rounding and by at most an iteration at
the stop: FP64 to 50 tol relative, FP32 vectors to 2e-5 (the bounds of the other parity
tests); seed solutions enter the gradient linearly, at the same bounds.
"""
import numpy as np
import pytest

import paper_1105_5256_gb300 as L
import synth

pytestmark = pytest.mark.gpu

K = {5: L.LD_STENCIL_2D5, 13: L.LD_STENCIL_2D13_SQ, 7: L.LD_STENCIL_3D7}
CASES = [
    # points, dims, periodic, kappa2, distance, form, gradient ids, shifts
    (5, (1, 40), False, 0.5, 2, "", (), 16),               # one column of vertices
    (5, (5, 3), True, 0.5, 1, "mask", (0, 1), 16),         # wraps within one CTA, partial item
    (13, (6, 5), True, 0.5, 1, "", (2,), 16),              # two halo lines that wrap onto own lines
    (13, (33, 7), False, 0.4, 1, "", (), 40),              # more shifts than a warp has lanes
    (5, (127, 61), False, 0.3, 2, "field", (0, 2), 20),
    (13, (126, 61), True, 0.3, 1, "", (0, 2), 20),         # torus ghosts in a partial item
    (13, (130, 90), False, 0.2, 2, "", (), 20),
    (5, (400, 260), True, 0.3, 4, "mask", (1,), 20),       # several CTAs a vector, mask bits
    (5, (1030, 12), False, 0.4, 2, "field", (0,), 20),     # wide lines: 258 groups of four
    (13, (301, 203), False, 0.3, 2, "", (0, 2), 20),
    (7, (9, 8, 7), True, 0.4, 2, "field", (0,), 20),
    (7, (21, 20, 19), False, 0.4, 2, "mask", (1, 2), 20),
    (7, (40, 33, 35), False, 0.4, 2, "", (), 20),
]


def build(case, prec, engine, col, tol, **kw):
    points, dims, per, k2, d, form, _, shifts = case
    n = int(np.prod(dims))
    field = synth.kappa2_field(7, dims) if form == "field" else None
    mask = synth.obs_mask(8, n, 0.2) if form == "mask" else None
    m = L.grid_matrix(K[points], dims, 1.0 if form == "field" else k2, periodic=per, kappa2_field=field,
                      tau=3.0 if form == "mask" else 0.0, obs_mask=mask, scale=1.7)
    return L.ld_create(m, d, shifts, tol, L.options(precision=prec, engine=engine, colouring=col, **kw))


def evaluate(ctx, ids):
    if ids:
        v, g, info = L.ld_logdet_grad(ctx, list(ids))
    else:
        (v, info), g = L.ld_logdet(ctx), np.zeros(0)
    return v, g, info, *L.ld_column_terms(ctx)


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "%d-%s%s%s" % (c[0], "x".join(map(str, c[1])), "t" if c[2] else "", c[5]))
def test_resident_matches_streaming_engine(case, prec):
    points, dims, per, k2, d, form, ids, shifts = case
    tol = 1e-9 if prec == L.LD_FP64 else 1e-6
    col, _ = L.ld_colour_grid(K[points], dims, per, d)
    ref = evaluate(build(case, prec, 1, col, tol, tile_width=2), ids)
    ctx = build(case, prec, 0, col, tol, tile_width=2)
    got = evaluate(ctx, ids)
    # FP64 lattices large enough to keep every SM's FP64 units busy either way may stream
    assert ref[2]["engine"] == 1 and (got[2]["engine"] == 4 or (prec == L.LD_FP64 and np.prod(dims) > 12000))
    bar = 50 * tol if prec == L.LD_FP64 else 2e-5
    for k in (3, 4):                                       # per-colour terms, seed projections
        err = np.linalg.norm(got[k] - ref[k]) / np.linalg.norm(ref[k])
        assert err <= bar, (k, err)
    assert abs(got[0] - ref[0]) <= bar * np.abs(ref[3]).sum()
    assert np.allclose(got[1], ref[1], rtol=bar, atol=0)
    assert abs(got[2]["iters"] - ref[2]["iters"]) <= max(3, ref[2]["iters"] // 10)
    if ids and prec == L.LD_FP64:                          # (in FP32 both are rounding, eps x condition)
        assert 0 <= got[2]["rel_resid_max"] <= 2 * max(tol, ref[2]["rel_resid_max"])
    again = evaluate(ctx, ids)                             # the same bits on every call
    assert again[0] == got[0] and np.array_equal(again[3], got[3]) and np.array_equal(again[1], got[1])


def test_partial_colour_ranges_keep_each_column():
    case = (13, (130, 90), False, 0.2, 2, "", (), 20)
    col, nc = L.ld_colour_grid(K[13], case[1], False, 2)
    ctx = build(case, L.LD_FP64, 0, col, 1e-8)
    whole, info = L.ld_logdet(ctx)
    assert info["engine"] == 4
    terms, _ = L.ld_column_terms(ctx)
    parts = [L.ld_logdet_partial(ctx, a, b)[0] for a, b in ((0, 5), (5, 5), (5, nc))]
    assert parts[1] == 0.0 and abs(sum(parts) - whole) <= 1e-13 * np.abs(terms).sum()


def test_partial_ranges_leave_zero_seed_solutions_elsewhere():
    """ld_grad after a partial solve sums over the colours of the range alone."""
    case = (5, (127, 61), False, 0.3, 2, "mask", (), 20)
    col, nc = L.ld_colour_grid(K[5], case[1], False, 2)
    grads = []
    for engine in (1, 0):
        ctx = build(case, L.LD_FP64, engine, col, 1e-10, keep_x0=1)
        L.ld_logdet(ctx)                                   # every colour's x on the device
        L.ld_logdet_partial(ctx, 2, nc - 1)
        grads.append(L.ld_grad(ctx, [L.LD_P_TAU, L.LD_P_SCALE]))
    assert np.allclose(grads[0], grads[1], rtol=50e-10, atol=0)


def test_iteration_cap_and_new_parameters():
    case = (5, (127, 61), False, 1e-4, 2, "", (), 20)
    col, _ = L.ld_colour_grid(K[5], case[1], False, 2)
    ctx = build(case, L.LD_FP64, 0, col, 1e-10, max_iter=20)
    with pytest.raises(L.LogDetError) as e:
        L.ld_logdet(ctx)
    assert e.value.status == L.LD_ENOTCONV
    L.ld_set_params(ctx, 50.0, 0.0, 1.7)                   # well conditioned: converges within the cap
    v, info = L.ld_logdet(ctx)
    other = build((5, (127, 61), False, 50.0, 2, "", (), 20), L.LD_FP64, 1, col, 1e-10)
    w, _ = L.ld_logdet(other)
    assert info["engine"] == 4 and abs(v - w) <= 50e-10 * abs(w)


# ------------------------------------------------------------------ CSR
def csr_problem(name):
    if name.startswith("mesh"):                            # mesh<alpha>-<nx>x<ny>
        alpha, size = name[4:].split("-")
        nx, ny = map(int, size.split("x"))
        p, t = synth.perturbed_triangulation(6, nx, ny)
        from paper_1105_5256_gb300 import mesh
        rp, ci, vv = mesh.spde_csr(p, t, 0.3 * (nx - 1) * (ny - 1), int(alpha), 1.0)
    else:
        n = int(name[4:])
        rp, ci, vv = synth.csr_from_edges(n, *synth.random_sparse_spd_pattern(9, n), 0.3)
    lo, hi, _ = *L.ld_csr_bounds(rp, ci, vv), None
    return rp, ci, vv, lo, hi


@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
@pytest.mark.parametrize("name,shifts", [
    ("rand9", 16),                # fewer rows than a warp, one or two a CTA
    ("rand333", 40),              # more shifts than lanes
    ("rand3001", 20),
    ("mesh1-31x27", 20),
    ("mesh2-40x33", 20),          # long rows, external columns on both sides
    ("mesh2-141x97", 20),         # several vectors a team and a remainder
])
def test_resident_csr_matches_streaming_engine(name, shifts, prec):
    rp, ci, vv, lo, hi = csr_problem(name)
    tol = 1e-9 if prec == L.LD_FP64 else 1e-6
    out = []
    for engine in (1, 0):
        ctx = L.ld_create(L.csr_matrix(rp, ci, vv, scale=1.3), 2, shifts, tol,
                          L.options(precision=prec, engine=engine, lambda_min=1.3 * lo, lambda_max=1.3 * hi, tile_width=2))
        out.append((ctx, evaluate(ctx, (L.LD_P_SCALE,))))
    ref, got = out[0][1], out[1][1]
    assert ref[2]["engine"] == 1 and got[2]["engine"] == 4
    bar = 50 * tol if prec == L.LD_FP64 else 2e-5
    for k in (3, 4):
        assert np.linalg.norm(got[k] - ref[k]) <= bar * np.linalg.norm(ref[k])
    assert np.allclose(got[1], ref[1], rtol=bar, atol=0)
    ctx = out[1][0]
    again = evaluate(ctx, (L.LD_P_SCALE,))
    assert again[0] == got[0] and np.array_equal(again[3], got[3]) and np.array_equal(again[1], got[1])
    nc = len(got[3])                                       # each column alike in any range
    split = [L.ld_logdet_partial(ctx, a, b)[0] for a, b in ((0, nc // 3), (nc // 3, nc))]
    assert abs(sum(split) - got[0]) <= 1e-13 * np.abs(got[3]).sum()


def test_resident_csr_reports_not_spd():
    n = 600
    rp, ci, vv = synth.csr_from_edges(n, *synth.random_sparse_spd_pattern(9, n), 0.3)
    ctx = L.ld_create(L.csr_matrix(rp, ci, -vv), 1, 16, 1e-8, L.options(lambda_min=0.1, lambda_max=50.0))
    with pytest.raises(L.LogDetError) as e:
        L.ld_logdet(ctx)
    assert e.value.status == L.LD_ENOTSPD


# ------------------------------------------------------------------ vector form
@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
@pytest.mark.parametrize("points,dims,per,form,ncols,shifts", [
    (5, (1, 9), False, "", 1, 16),
    (5, (33, 21), True, "mask", 3, 40),       # more shifts than a warp has lanes
    (5, (62, 51), False, "field", 5, 20),
    (13, (30, 34), True, "", 4, 20),          # one CTA a column, torus ghosts
    (13, (130, 90), False, "", 2, 20),        # teams of many CTAs
    (13, (48, 40), False, "", 160, 20),       # more columns than SMs
    (7, (13, 11, 10), False, "field", 3, 20),
])
def test_resident_vector_form_matches_streaming_engine(points, dims, per, form, ncols, shifts, prec):
    """log(Q) V and Q^{-1/2} V: the coefficient form on chip against the shifted directions.
    Both stop each shift at a relative residual tol: 50 tol relative (FP32 vectors: 2e-5)."""
    tol = 1e-9 if prec == L.LD_FP64 else 1e-6
    n = int(np.prod(dims))
    V = synth.random_probe_block(3, n, ncols)
    V[:, -1] = 0.0 if ncols > 1 else V[:, -1]              # a zero column stays zero
    out = []
    for engine in (1, 0):
        ctx = build((points, dims, per, 0.3, 1, form, (), shifts), prec, engine, None, tol)
        Y, info = L.ld_logmv(ctx, V)
        Z, _ = L.ld_invsqrt_mv(ctx, V)
        out.append((Y, Z, info, L.ld_logmv(ctx, V)[0]))
    assert out[0][2]["engine"] != 4 and out[1][2]["engine"] == 4
    bar = 50 * tol if prec == L.LD_FP64 else 2e-5
    for k in (0, 1):
        assert np.linalg.norm(out[1][k] - out[0][k]) <= bar * np.linalg.norm(out[0][k])
    assert np.array_equal(out[1][0], out[1][3])
    if ncols > 1:
        assert not out[1][0][:, -1].any()


def test_vector_form_errors_leave_the_context_usable():
    V = synth.random_probe_block(3, 40 * 30, 2)
    ctx = build((5, (40, 30), False, 1e-4, 1, "", (), 20), L.LD_FP64, 0, None, 1e-10, max_iter=20)
    Y = np.zeros_like(V)
    with pytest.raises(L.LogDetError) as e:
        L.ld_logmv(ctx, V)
    assert e.value.status == L.LD_ENOTCONV
    L.ld_set_params(ctx, 50.0, 0.0, 1.7)
    Y, info = L.ld_logmv(ctx, V)
    W, _ = L.ld_logmv(build((5, (40, 30), False, 50.0, 1, "", (), 20), L.LD_FP64, 1, None, 1e-10), V)
    assert info["engine"] == 4 and np.linalg.norm(Y - W) <= 50e-10 * np.linalg.norm(W)


# ------------------------------------------------------------------ batches
@pytest.mark.parametrize("prec", [L.LD_FP64, L.LD_MIXED])
def test_resident_batch_matches_single_solves(prec):
    """A batch over kinds, boundaries and sizes from one CTA a column to sixteen, and a lattice
    too wide for any cluster beside them, against streaming contexts one by one (both stop at
    tol: 50 tol of the terms' sum, FP32 vectors 2e-5)."""
    tol = 1e-9 if prec == L.LD_FP64 else 1e-6
    insts = [(5, (9, 7), False, 0.5, 2, ""), (13, (30, 34), True, 0.3, 1, ""), (5, (61, 50), True, 0.3, 2, "mask"),
             (7, (13, 11, 10), False, 1.0, 2, "field"), (13, (130, 90), False, 0.2, 2, ""), (5, (300, 220), False, 0.5, 1, ""),
             (5, (2100, 6), False, 0.5, 1, ""), (13, (200, 210), False, 0.6, 1, "")]
    mats, ref, bars = [], [], []
    for points, dims, per, k2, d, form in insts:
        n = int(np.prod(dims))
        m = lambda: L.grid_matrix(K[points], dims, k2, periodic=per, tau=3.0 if form == "mask" else 0.0,
                                  kappa2_field=synth.kappa2_field(7, dims) if form == "field" else None,
                                  obs_mask=synth.obs_mask(8, n, 0.2) if form == "mask" else None)
        mats.append(m())
        ctx = L.ld_create(m(), d, 20, tol, L.options(precision=prec, engine=1, tile_width=2))
        ref.append(L.ld_logdet(ctx)[0])
        bars.append((50 * tol if prec == L.LD_FP64 else 2e-5) * np.abs(L.ld_column_terms(ctx)[0]).sum())
    b = L.ld_batch_create(mats, [i[4] for i in insts], 20, tol, L.options(precision=prec))
    vals, grads, info = L.ld_batch_logdet(b, with_grad=True)
    assert np.all(np.abs(vals - ref) <= bars), (vals, ref)
    assert np.isnan(grads[1]) and np.isnan(grads[3]) and np.all(np.isfinite(np.delete(grads, [1, 3, 4, 7])))
    again, _, _ = L.ld_batch_logdet(b)
    assert np.array_equal(again, vals)


def test_resident_batch_names_the_instance_that_fails():
    mats = [L.grid_matrix(K[5], (40, 30), k2) for k2 in (0.5, 1e-5, 0.5)]
    b = L.ld_batch_create(mats, [1, 1, 1], 20, 1e-10, L.options(max_iter=60))
    with pytest.raises(L.LogDetError) as e:
        L.ld_batch_logdet(b)
    assert e.value.status == L.LD_ENOTCONV and "instance 1" in str(e.value)
