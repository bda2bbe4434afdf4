"""Workloads of the log-determinant library over the range it is used in.

A case is one evaluation as a fitting or prediction program makes it: the context (matrix,
colouring, device buffers) exists, new hyperparameters arrive, and the call returns the log
det and what the option asks for beside it.  Families:

  grid       ld_set_params + ld_logdet / ld_logdet_grad on a lattice precision (5-point,
             13-point Matern or 7-point; scalar kappa^2, a kappa^2 field or a mask)
  likelihood one call of fit.Likelihood (log det, gradient and the quadratic forms)
  torus_csr  ld_logdet on a torus given as a CSR matrix
  mesh       ld_logdet on a finite-element precision of a triangulation (CSR)
  batch      ld_batch_logdet on many independent lattices of uneven size
  sample     ld_invsqrt_mv: draws x = Q^{-1/2} z from given normal z

Mixed-precision contexts keep their vectors in FP32, so their results are returned as FP32;
FP64 contexts return FP64.  exact() computes the same probed quantities from closed-form
eigenvalues (lattices with a scalar kappa^2) or from FP64 CG with the Gauss quadrature of
its tridiagonal matrix, in torch and numpy alone.
"""
import math

import numpy as np
import torch

import paper_1105_5256_gb300 as L
from paper_1105_5256_gb300 import fit, mesh

KINDS = {5: L.LD_STENCIL_2D5, 13: L.LD_STENCIL_2D13_SQ, 7: L.LD_STENCIL_3D7}
PARAMS = {"kappa2": L.LD_P_KAPPA2, "tau": L.LD_P_TAU, "scale": L.LD_P_SCALE}


def _grid(name, points, nx, ny, nz=1, kappa2=0.1, precision="mixed", distance=2, shifts=20, tol=1e-6,
          periodic=False, field=False, tau=0.0, grad="", reliable=0.0):
    c = {"family": "grid", "points": points, "nx": nx, "ny": ny, "nz": nz, "kappa2": kappa2,
         "precision": precision, "distance": distance, "shifts": shifts, "tol": tol, "periodic": periodic,
         "field": field, "tau": tau, "grad": grad, "reliable": reliable}
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest call: a 64^2 torus handed over as CSR, FP64, latency-bound.
        {"name": "torus_csr_64_fp64", "family": "torus_csr", "nx": 64, "ny": 64, "kappa2": 0.5, "precision": "fp64",
         "distance": 4, "shifts": 20, "tol": 1e-10},
        # One step of a maximum-likelihood fit on a small field (default FP64): called hundreds
        # of times by the Newton iteration.
        {"name": "likelihood_48x40_fp64", "family": "likelihood", "points": 13, "nx": 48, "ny": 40, "kappa2": 0.1,
         "samples": 4, "distance": 4, "shifts": 20, "tol": 1e-9},
        # Gauss-linear posterior with an observation mask, FP64, with both gradients.
        _grid("posterior_128_fp64", 5, 128, 128, kappa2=0.1, precision="fp64", distance=4, tol=1e-10, tau=4.0,
              grad="kappa2,tau"),
        # An ordinary Matern field of odd shape with the gradient a fit needs, mixed precision.
        _grid("matern_300x200_grad", 13, 300, 200, kappa2=0.1, grad="kappa2,scale"),
        # The default options (FP64) on a larger Matern field.
        _grid("matern_512x384_fp64", 13, 512, 384, kappa2=0.2, precision="fp64"),
        # A non-stationary field on a torus (global or cylindrical domains), with its gradient.
        _grid("torus_field_500x333_grad", 5, 500, 333, kappa2=1.0, distance=4, periodic=True, field=True,
              grad="kappa2"),
        # The headline workload: Matern precision on a 1024^2 grid, mixed precision.
        _grid("matern_1024", 13, 1024, 1024, kappa2=0.1),
        # The largest lattice: a 2048^2 posterior with reliable updates and both gradients.
        _grid("posterior_2048_grad", 5, 2048, 2048, kappa2=0.1, distance=4, tol=1e-9, tau=4.0, grad="kappa2,tau",
              reliable=1e-2),
        # A 3D non-stationary field with the gradient of its scale.
        _grid("field_3d_128_grad", 7, 128, 128, 128, kappa2=1.0, distance=6, shifts=32, field=True, grad="kappa2"),
        # A general mesh through finite elements (CSR), mixed precision.
        {"name": "mesh_320x280", "family": "mesh", "nx": 320, "ny": 280, "alpha": 2, "kappa2": 0.1,
         "precision": "mixed", "distance": 2, "shifts": 20, "tol": 1e-6, "mesh_seed": 6},
        # Many independent fields of uneven size evaluated at once.
        {"name": "batch_64", "family": "batch", "count": 64, "side_lo": 32, "side_hi": 512, "shape_seed": 3,
         "kappa2_lo": 0.03, "kappa2_hi": 1.0, "precision": "mixed", "shifts": 20, "tol": 1e-6},
        # Simulation of fields: four draws of a Matern field at once, FP64.
        {"name": "sample_200x150_fp64", "family": "sample", "points": 13, "nx": 200, "ny": 150, "kappa2": 0.1,
         "samples": 4, "shifts": 24, "tol": 1e-10},
    ]


def draw(rng):
    """One more case of the listed families: sizes log-uniform over the range, odd ones among them."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def k2(lo, hi):
        return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    f = rng.choice(["grid", "grid", "grid", "grid", "grid", "grid", "likelihood", "torus_csr", "mesh", "batch",
                    "sample"])
    if f == "torus_csr":
        return {"family": f, "nx": size(24, 100), "ny": size(24, 100), "kappa2": k2(0.1, 1.0), "precision": "fp64",
                "distance": rng.choice([2, 4]), "shifts": 20, "tol": 1e-10}
    if f == "likelihood":
        return {"family": f, "points": rng.choice([5, 13]), "nx": size(24, 96), "ny": size(24, 96),
                "kappa2": k2(0.1, 1.0), "samples": rng.randint(1, 8), "distance": rng.choice([2, 4]), "shifts": 20,
                "tol": 1e-9}
    if f == "sample":
        return {"family": f, "points": rng.choice([5, 13]), "nx": size(32, 220), "ny": size(32, 220),
                "kappa2": k2(0.1, 1.0), "samples": rng.randint(1, 6), "shifts": 24, "tol": 1e-10}
    if f == "mesh":
        return {"family": f, "nx": size(32, 320), "ny": size(32, 280), "alpha": rng.choice([1, 2]),
                "kappa2": k2(0.1, 1.0), "precision": rng.choice(["mixed", "fp64"]), "distance": 2, "shifts": 20,
                "tol": 1e-6, "mesh_seed": rng.randint(0, 999)}
    if f == "batch":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        return {"family": f, "count": rng.randint(8, 48), "side_lo": 32,
                "side_hi": size(64, 512 if precision == "mixed" else 160), "shape_seed": rng.randint(0, 999),
                "kappa2_lo": 0.05, "kappa2_hi": 1.0, "precision": precision, "shifts": 20, "tol": 1e-6}
    points = rng.choice([5, 13, 5, 13, 7])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    periodic = rng.random() < 0.25
    if points == 7:
        field = rng.random() < 0.5
        # a scalar kappa^2 of a small FP64 3D grid, or a mixed one up to the listed size
        hi = 128 if precision == "mixed" else 48
        return _grid(None, 7, size(16, hi), size(16, hi), size(16, hi), kappa2=1.0 if field else k2(0.1, 1.0),
                     precision=precision, distance=4, shifts=20, tol=1e-6, periodic=periodic, field=field,
                     grad=rng.choice(["", "kappa2"]))
    hi = 440 if precision == "fp64" else 1024 if points == 13 else 2048
    if periodic:
        hi = min(hi, 512)
    nx, ny = size(48, hi), size(48, hi)
    # ill-conditioned Matern fields only where the grid is small enough for the range's cost
    kk = k2(0.05, 1.0) if points == 5 else k2(0.1 if precision == "mixed" else 0.2, 1.0)
    if points == 13:
        return _grid(None, 13, nx, ny, kappa2=kk, precision=precision, distance=rng.choice([1, 2]),
                     periodic=periodic, grad=rng.choice(["", "", "kappa2,scale"]))
    form = rng.choice(["scalar", "field", "mask"])
    tol = rng.choice([1e-6, 1e-8])
    reliable = 1e-2 if precision == "mixed" and form == "mask" else 0.0
    if form == "scalar":
        return _grid(None, 5, nx, ny, kappa2=kk, precision=precision, distance=4, tol=tol, periodic=periodic,
                     grad=rng.choice(["", "kappa2"]))
    if form == "field":
        return _grid(None, 5, nx, ny, kappa2=1.0, precision=precision, distance=4, tol=tol, periodic=periodic,
                     field=True, grad=rng.choice(["", "kappa2"]))
    return _grid(None, 5, nx, ny, kappa2=kk, precision=precision, distance=4, tol=1e-9, periodic=periodic, tau=4.0,
                 grad=rng.choice(["", "kappa2,tau"]), reliable=reliable)


# ------------------------------------------------------------------ inputs from a seed
def _kappa2(case, seed):
    """The hyperparameter an optimiser would ask for: within 5 % of the case's."""
    return float(case["kappa2"] * (1.0 + 0.1 * (np.random.default_rng(seed).random() - 0.5)))


def _dims(case):
    return (case["nx"], case["ny"]) if case.get("nz", 1) == 1 and case.get("points") != 7 else (
        case["nx"], case["ny"], case["nz"])


def _field(case, seed):
    """kappa^2(s): log-normal, smoothed by a 5-wide truncated box mean (mean -2, sd 1 of its log)."""
    z = np.random.default_rng([seed, 1]).standard_normal(tuple(reversed(_dims(case))))
    for ax in range(z.ndim):
        c = np.concatenate([np.zeros_like(np.take(z, [0], axis=ax)), np.cumsum(z, axis=ax)], axis=ax)
        i = np.arange(z.shape[ax])
        hi, lo = np.minimum(i + 3, z.shape[ax]), np.maximum(i - 2, 0)
        shape = [1] * z.ndim
        shape[ax] = -1
        z = (np.take(c, hi, axis=ax) - np.take(c, lo, axis=ax)) / (hi - lo).reshape(shape)
    return np.exp(-2.0 + (z - z.mean()) / z.std()).reshape(-1)


def _mask(case, seed):
    """A tenth of the nodes observed."""
    n = int(np.prod(_dims(case)))
    m = np.zeros(n, dtype=np.uint8)
    m[np.random.default_rng([seed, 2]).permutation(n)[: round(0.1 * n)]] = 1
    return m


def _torus_csr(nx, ny, kappa2):
    i = np.arange(nx * ny).reshape(ny, nx)
    cols = np.stack([i, np.roll(i, 1, 0), np.roll(i, -1, 0), np.roll(i, 1, 1), np.roll(i, -1, 1)]).reshape(5, -1).T
    vals = np.broadcast_to(np.array([kappa2 + 4.0, -1.0, -1.0, -1.0, -1.0]), cols.shape)
    order = np.argsort(cols, axis=1)
    rowptr = np.arange(0, 5 * nx * ny + 1, 5, dtype=np.int64)
    return (rowptr, np.take_along_axis(cols, order, 1).reshape(-1).astype(np.int32),
            np.take_along_axis(vals, order, 1).reshape(-1).copy())


def _triangulation(case):
    """Vertices of an nx x ny lattice on the unit square moved by up to 0.15 spacings, cells cut at random."""
    nx, ny = case["nx"], case["ny"]
    g = np.random.default_rng([case["mesh_seed"], 3])
    ix, iy = (a.ravel() for a in np.meshgrid(np.arange(nx), np.arange(ny)))
    dx, dy = g.uniform(-0.15, 0.15, ix.size), g.uniform(-0.15, 0.15, ix.size)
    dx[(ix == 0) | (ix == nx - 1)] = 0.0
    dy[(iy == 0) | (iy == ny - 1)] = 0.0
    pts = np.stack([(ix + dx) / (nx - 1), (iy + dy) / (ny - 1)], axis=1)
    cx, cy = np.meshgrid(np.arange(nx - 1), np.arange(ny - 1))
    a = (cx + nx * cy).ravel()
    b, c, d = a + 1, a + nx, a + nx + 1
    coin = g.integers(0, 2, size=(a.size, 1)).astype(bool)
    return pts, np.concatenate([np.where(coin, np.stack([a, b, d], 1), np.stack([a, b, c], 1)),
                                np.where(coin, np.stack([a, d, c], 1), np.stack([b, d, c], 1))]).astype(np.int64)


def _mesh_kappa2(case, seed):
    """kappa^2 on the unit square such that kappa^2 h^2 is the case's lattice value."""
    return _kappa2(case, seed) * (math.sqrt(case["nx"] * case["ny"]) - 1.0) ** 2


def _lumped(pts, tri):
    e1, e2 = pts[tri[:, 1]] - pts[tri[:, 0]], pts[tri[:, 2]] - pts[tri[:, 0]]
    area = 0.5 * np.abs(e1[:, 0] * e2[:, 1] - e1[:, 1] * e2[:, 0])
    return np.bincount(tri.ravel(), weights=np.repeat(area / 3.0, 3), minlength=pts.shape[0]), area


def _batch_shapes(case):
    """(points, side) of every lattice of a batch."""
    g = np.random.default_rng([case["shape_seed"], 4])
    sides = g.integers(case["side_lo"], case["side_hi"] + 1, size=case["count"])
    return [(5 if p else 13, int(s)) for p, s in zip(g.integers(0, 2, size=case["count"]), sides)]


def _batch_kappa2(case, seed):
    g = np.random.default_rng([case["shape_seed"], 5])
    base = np.exp(g.uniform(math.log(case["kappa2_lo"]), math.log(case["kappa2_hi"]), size=case["count"]))
    return base * (1.0 + 0.1 * (np.random.default_rng(seed).random(case["count"]) - 0.5))


def _normals(case, seed):
    return np.random.default_rng([seed, 6]).standard_normal((int(np.prod(_dims(case))), case["samples"]))


_stored = {}


def _colouring(case):
    """The greedy colouring of a lattice, computed once per shape and stored, as the method prescribes."""
    key = (case["points"], _dims(case), case["periodic"], case["distance"])
    if key not in _stored:
        _stored[key] = L.ld_colour_grid(KINDS[case["points"]], _dims(case), case["periodic"], case["distance"])[0]
    return _stored[key]


def _precision(case):
    return L.LD_MIXED if case["precision"] == "mixed" else L.LD_FP64


# ------------------------------------------------------------------ one case
def prepare(case, seed):
    f = case["family"]
    state = {"case": case}
    if f == "grid":
        grad = [PARAMS[p] for p in case["grad"].split(",") if p]
        opts = L.options(precision=_precision(case), colouring=_colouring(case), reliable_delta=case["reliable"])
        m = L.grid_matrix(KINDS[case["points"]], _dims(case), case["kappa2"], periodic=case["periodic"],
                          kappa2_field=_field(case, seed) if case["field"] else None, tau=case["tau"],
                          obs_mask=_mask(case, seed) if case["tau"] > 0 else None)
        state.update(ctx=L.ld_create(m, case["distance"], case["shifts"], case["tol"], opts), grad=grad,
                     params=(_kappa2(case, seed), case["tau"], 1.0))
    elif f == "likelihood":
        y = _normals(case, seed) / 4.0
        state.update(lik=fit.Likelihood(KINDS[case["points"]], _dims(case), y, case["distance"],
                                        n_shifts=case["shifts"], tol=case["tol"]),
                     eta=np.log([_kappa2(case, seed), 1.3]))
    elif f == "torus_csr":
        k2 = _kappa2(case, seed)
        state["ctx"] = L.ld_create(L.csr_matrix(*_torus_csr(case["nx"], case["ny"], k2)), case["distance"],
                                   case["shifts"], case["tol"],
                                   L.options(precision=_precision(case), lambda_min=k2, lambda_max=k2 + 8.0))
    elif f == "mesh":
        pts, tri = _triangulation(case)
        k2 = _mesh_kappa2(case, seed)
        rowptr, col, val = mesh.spde_csr(pts, tri, k2, case["alpha"])
        c = _lumped(pts, tri)[0]
        lo = k2 * k2 * c.min() ** 2 / c.max() if case["alpha"] == 2 else k2 * c.min()
        hi = float(np.add.reduceat(np.abs(val), rowptr[:-1]).max())
        state["ctx"] = L.ld_create(L.csr_matrix(rowptr, col, val), case["distance"], case["shifts"], case["tol"],
                                   L.options(precision=_precision(case), lambda_min=lo, lambda_max=hi))
    elif f == "batch":
        shapes = _batch_shapes(case)
        mats = [L.grid_matrix(KINDS[p], (s, s), k) for (p, s), k in zip(shapes, _batch_kappa2(case, seed))]
        state["ctx"] = L.ld_batch_create(mats, [4 if p == 5 else 2 for p, _ in shapes], case["shifts"], case["tol"],
                                         L.options(precision=_precision(case)))
    else:
        m = L.grid_matrix(KINDS[case["points"]], _dims(case), _kappa2(case, seed))
        state.update(ctx=L.ld_create(m, 1, case["shifts"], case["tol"], L.options(precision=L.LD_FP64)),
                     z=_normals(case, seed))
    return state


def run(state):
    case = state["case"]
    f = case["family"]
    if f == "likelihood":
        value, grad = state["lik"](state["eta"])
        return {"value": np.float64(value), "grad": np.asarray(grad)}
    if f == "sample":
        return {"x": L.ld_invsqrt_mv(state["ctx"], state["z"])[0]}
    real = np.float32 if case["precision"] == "mixed" else np.float64
    if f == "batch":
        values, grads, _ = L.ld_batch_logdet(state["ctx"], with_grad=True)
        return {"logdet": values.astype(real), "grad": grads.astype(real)}
    ctx = state["ctx"]
    if f == "grid":
        L.ld_set_params(ctx, *state["params"])
        if state["grad"]:
            value, grad, _ = L.ld_logdet_grad(ctx, state["grad"])
            return {"logdet": real(value), "grad": grad.astype(real)}
    value, _ = L.ld_logdet(ctx)
    terms, seeds = L.ld_column_terms(ctx)
    return {"logdet": real(value), "terms": terms.astype(real), "seeds": seeds.astype(real)}


# ------------------------------------------------------------------ work
def _iterations(points, dim, kappa2, tol, tau=0.0):
    """CG's bound sqrt(cond)/2 log(2/tol) for the lattice operator."""
    cond = (kappa2 + 4.0 * dim + tau) / kappa2
    return 0.5 * (cond if points == 13 else math.sqrt(cond)) * math.log(2.0 / tol)


# flops a vertex and column of one CG step: the two updates, the three dot products of CG
# and one indicator product, and the operator (5-, 13- or 7-point as its square root twice)
_FLOPS = {5: 4 + 7 + 7, 13: 4 + 7 + 14, 7: 4 + 7 + 9}


def _colours(points, distance):
    """Vertices within the colouring's reach that are mutually that close: the classes any colouring needs."""
    d = distance * (2 if points == 13 else 1)
    if points == 7:
        return (d + 1) * (d * d / 2 + d + 3) / 3
    return ((d + 1) ** 2 + 1) // 2


def work(case):
    """One pass: the per-vertex inputs (colours, kappa^2 field, mask, matrix, right-hand sides) read
    once and the results written; the flops of CG on every probing vector."""
    f = case["family"]
    if f == "batch":
        n = it = 0.0
        for (p, s), k in zip(_batch_shapes(case), _batch_kappa2(case, 0)):
            n += s * s
            it += s * s * _colours(p, 4 if p == 5 else 2) * _iterations(p, 2, k, case["tol"]) * _FLOPS[p]
        return {"bytes": 4.0 * n + 16.0 * case["count"], "flops": float(it)}
    points = case.get("points", 5)
    if f == "mesh":
        points = 5 if case["alpha"] == 1 else 13
    n = case["nx"] * case["ny"] * case.get("nz", 1)
    dim = 3 if points == 7 else 2
    kappa2 = 0.05 if case.get("field") else case["kappa2"]
    it = _iterations(points, dim, kappa2, case["tol"], case.get("tau", 0.0))
    cols = case["samples"] if f == "sample" else _colours(points, case["distance"])
    flops = _FLOPS[points] * n * cols * it
    data = 4.0 * n + 8.0 * cols
    if f == "sample":
        data = 16.0 * n * case["samples"]
        flops += 12.0 * case["shifts"] * n * cols * it       # complex update of every shifted direction
    elif f == "likelihood":
        data += 8.0 * n * case["samples"]
    elif f in ("torus_csr", "mesh"):
        per_row = 5 if f == "torus_csr" else 7 if case["alpha"] == 1 else 19
        word = 4 if case["precision"] == "mixed" else 8
        data += n * (8.0 + per_row * (4.0 + word))
        flops += 2.0 * (per_row - points) * n * cols * it
    else:
        data += n * ((8.0 if case["field"] else 0.0) + (1.0 if case["tau"] > 0 else 0.0))
    return {"bytes": data, "flops": flops}


# ------------------------------------------------------------------ exact values in 64 bits
def _greedy(n, near):
    """Smallest free colour in natural order; near(i) yields the vertices within the distance."""
    colour = [-1] * n
    for i in range(n):
        used = 0
        for j in near(i):
            if j < i:
                used |= 1 << colour[j]
        colour[i] = (~used & (used + 1)).bit_length() - 1
    return np.array(colour)


def _lattice_colours(points, dims, periodic, distance):
    """Greedy colouring of the lattice ball of radius d (2 d for the 13-point kind)."""
    r = distance * (2 if points == 13 else 1)
    dims = tuple(dims) + (1,) * (3 - len(dims))
    nx, ny, nz = dims
    rng = [range(-r, r + 1) if s > 1 else (0,) for s in dims]
    ball = [(dx, dy, dz) for dz in rng[2] for dy in rng[1] for dx in rng[0]
            if 0 < abs(dx) + abs(dy) + abs(dz) <= r]
    if periodic:
        def near(i):
            x, y, z = i % nx, i // nx % ny, i // (nx * ny)
            return [(x + a) % nx + nx * ((y + b) % ny + ny * ((z + c) % nz)) for a, b, c in ball]
        return _greedy(nx * ny * nz, near)
    # wavefronts x + a y + b z = t, on which no vertex is near another and all earlier ones are done
    before = np.array([o for o in ball if (o[2], o[1], o[0]) < (0, 0, 0)])
    a = r + 1
    b = a * r + 1
    out = np.full((nz + 2 * r, ny + 2 * r, nx + 2 * r), -1, dtype=np.int64)
    flat = out.reshape(-1)
    sy, sz = nx + 2 * r, (nx + 2 * r) * (ny + 2 * r)
    off = before[:, 0] + sy * before[:, 1] + sz * before[:, 2]
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    t = (x + a * y + b * z).reshape(-1)
    order = np.argsort(t, kind="stable")
    place = ((x + r) + sy * (y + r) + sz * (z + r)).reshape(-1)[order]
    starts = np.searchsorted(t[order], np.arange(t.max() + 2))
    most = len(off) + 2
    for k in range(len(starts) - 1):
        p = place[starts[k]:starts[k + 1]]
        if p.size == 0:
            continue
        used = np.zeros((p.size, most), dtype=bool)
        used[np.arange(p.size)[:, None], flat[p[:, None] + off]] = True      # -1 marks the last place
        flat[p] = np.argmin(used, axis=1)
    return out[r:r + nz, r:r + ny, r:r + nx].reshape(-1).copy()


def _dst(n):
    k = torch.arange(1, n + 1, dtype=torch.float64)
    return (math.sqrt(2.0 / (n + 1)) * torch.sin(torch.outer(k, k) * (math.pi / (n + 1)))).cuda()


def _eigen(dims, periodic):
    """Eigenvalues of -Lap on the lattice, shaped (nz, ny, nx)."""
    lam = torch.zeros(1, 1, 1, dtype=torch.float64, device="cuda")
    for ax, n in enumerate(tuple(dims) + (None,) * (3 - len(dims))):
        if n is None:
            continue
        k = torch.arange(n, dtype=torch.float64, device="cuda")
        a = (2 - 2 * torch.cos(2 * math.pi * k / n)) if periodic else (2 - 2 * torch.cos(math.pi * (k + 1) / (n + 1)))
        lam = lam + a.reshape([-1 if i == 2 - ax else 1 for i in range(3)])
    return lam


def _transform(v, periodic):
    """Squared coefficients of v (nz, ny, nx) in the eigenvectors of the lattice Laplacian."""
    if periodic:
        return torch.fft.fftn(v).abs() ** 2 / v.numel()
    return _dst_apply(v) ** 2


def _dst_apply(v):
    v = v @ _dst(v.shape[2])
    v = torch.einsum("ab,zbx->zax", _dst(v.shape[1]), v)
    if v.shape[0] > 1:
        v = torch.einsum("ab,byx->ayx", _dst(v.shape[0]), v)
    return v


def _closed(points, dims, periodic, distance, kappa2, scale=1.0, colour=None):
    """Per colour: v^T log(Q) v, v^T Q^{-1} v, and d log det / d kappa^2 probed, scalar kappa^2."""
    if colour is None:
        colour = _lattice_colours(points, dims, periodic, distance)
    c = torch.from_numpy(np.asarray(colour)).cuda().reshape(tuple(reversed(tuple(dims) + (1,) * (3 - len(dims)))))
    q1 = kappa2 + _eigen(dims, periodic)
    q = scale * (q1 * q1 if points == 13 else q1)
    dq = scale * (2 * q1 if points == 13 else torch.ones_like(q1))
    terms, seeds, dk = [], [], []
    for k in range(int(c.max()) + 1):
        w = _transform((c == k).double(), periodic)
        terms.append((w * torch.log(q)).sum())
        seeds.append((w / q).sum())
        dk.append((w * dq / q).sum())
    return (torch.stack(a).cpu().numpy() for a in (terms, seeds, dk))


def _by_cg(apply, colour, tol=1e-12, most=6000):
    """Per colour v^T log(Q) v, v^T Q^{-1} v and the diagonal x_c[i] at the vertices i of class c, by
    FP64 CG and the Gauss quadrature of its tridiagonal matrix; apply acts on (n, C) blocks."""
    colour = torch.from_numpy(np.asarray(colour)).cuda()
    n, C = colour.numel(), int(colour.max()) + 1
    terms, seeds = np.zeros(C), np.zeros(C)
    own = torch.zeros(n, dtype=torch.float64, device="cuda")
    group = max(1, min(C, int(3e10 // (8 * n * 6))))
    for g0 in range(0, C, group):
        cols = torch.arange(g0, min(C, g0 + group), device="cuda")
        v = (colour[:, None] == cols[None, :]).double()
        vv = v.sum(0)
        r, p, x, rho = v.clone(), v.clone(), torch.zeros_like(v), vv.clone()
        al, be = [], []
        for it in range(most):
            w = apply(p)
            a = torch.where(rho > 0, rho / (p * w).sum(0).clamp_min(1e-300), 0)
            x.addcmul_(p, a.expand_as(p))
            r.addcmul_(w, -a.expand_as(w))
            new = (r * r).sum(0)
            b = torch.where(rho > 0, new / rho.clamp_min(1e-300), 0)
            al.append(a)
            be.append(b)
            rho = new
            p.mul_(b).add_(r)
            if it % 10 == 9 and bool((rho <= tol * tol * vv).all()):
                break
        a, b = torch.stack(al, 1), torch.stack(be, 1)
        k = a.shape[1]
        d = 1.0 / a
        d[:, 1:] += b[:, :-1] / a[:, :-1]
        o = b[:, :-1].sqrt() / a[:, :-1]
        for i in range(len(cols)):
            t = torch.diag(d[i]) + torch.diag(o[i], 1) + torch.diag(o[i], -1)
            lam, vec = torch.linalg.eigh(t)
            terms[g0 + i] = float(vv[i] * (vec[0] ** 2 * torch.log(lam)).sum())
        seeds[g0:g0 + len(cols)] = (v * x).sum(0).cpu().numpy()
        own += (v * x).sum(1)
        del v, r, p, x, w
    return terms, seeds, own


def _lattice_apply(dims, periodic, diag):
    """p -> diag p + sum over neighbours (p_i - p_j), Dirichlet ghosts zero; (n, C) blocks."""
    shape = tuple(reversed(tuple(dims)))

    def apply(p):
        q = p.reshape(shape + (p.shape[1],))
        w = (diag.reshape(shape + (1,)) + 2.0 * len(dims)) * q
        for ax in range(len(dims)):
            m = shape[ax]
            if periodic:
                w -= torch.roll(q, 1, ax)
                w -= torch.roll(q, -1, ax)
            else:
                w.narrow(ax, 1, m - 1).sub_(q.narrow(ax, 0, m - 1))
                w.narrow(ax, 0, m - 1).sub_(q.narrow(ax, 1, m - 1))
        return w.reshape(p.shape)
    return apply


def _fem(case, seed):
    """P1 finite-element precision of the case's mesh as a dense-index sparse tensor and its pattern."""
    pts, tri = _triangulation(case)
    k2 = _mesh_kappa2(case, seed)
    c, area = _lumped(pts, tri)
    # gradients of the barycentric coordinates: perpendicular to the opposite edge over twice the area
    rows, cols, vals = [], [], []
    edge = [pts[tri[:, (k + 2) % 3]] - pts[tri[:, (k + 1) % 3]] for k in range(3)]
    for a in range(3):
        for b in range(3):
            rows.append(tri[:, a])
            cols.append(tri[:, b])
            vals.append((edge[a] * edge[b]).sum(1) / (4.0 * area))
    n = pts.shape[0]
    d = np.arange(n)
    idx = torch.from_numpy(np.stack([np.concatenate(rows + [d]), np.concatenate(cols + [d])]))
    K = torch.sparse_coo_tensor(idx, torch.from_numpy(np.concatenate(vals + [k2 * c])), (n, n)).cuda().coalesce()
    Kc = K.to_sparse_csr()
    if case["alpha"] == 1:
        return (lambda p: torch.sparse.mm(Kc, p)), K
    inv = torch.from_numpy(1.0 / c).cuda()[:, None]
    return (lambda p: torch.sparse.mm(Kc, inv * torch.sparse.mm(Kc, p))), K


def _mesh_colours(K, alpha, distance):
    i, j = K.indices().cpu().numpy()
    n = K.shape[0]
    at = np.searchsorted(i, np.arange(n + 1))
    nbr = [j[at[k]:at[k + 1]].tolist() for k in range(n)]
    hops = distance * alpha

    def near(v):
        seen, edge = {v}, [v]
        for _ in range(hops):
            edge = {u for w in edge for u in nbr[w]} - seen
            seen |= edge
        seen.discard(v)
        return seen
    return _greedy(n, near)


def exact(case, seed):
    f = case["family"]
    if f == "torus_csr":
        t, s, _ = _closed(5, (case["nx"], case["ny"]), True, case["distance"], _kappa2(case, seed))
        return {"logdet": np.float64(t.sum()), "terms": t, "seeds": s}
    if f == "sample":
        q1 = _kappa2(case, seed) + _eigen(_dims(case), False)
        z = torch.from_numpy(_normals(case, seed)).cuda()
        root = q1 if case["points"] == 13 else q1.sqrt()
        x = torch.stack([_dst_apply(_dst_apply(z[:, k].reshape(root.shape)) / root).reshape(-1)
                         for k in range(z.shape[1])], dim=1)
        return {"x": x}
    if f == "likelihood":
        k2, s, S = _kappa2(case, seed), 1.3, case["samples"]
        t, _, dk = _closed(case["points"], _dims(case), False, case["distance"], k2, s)
        y = torch.from_numpy(_normals(case, seed) / 4.0).cuda()
        q1 = _lattice_apply(_dims(case), False, torch.full((y.shape[0],), k2, dtype=torch.float64, device="cuda"))
        u = q1(y)
        quad = float((u * u).sum() if case["points"] == 13 else (y * u).sum())      # y^T Q y / s
        dquad = float(2 * (y * u).sum() if case["points"] == 13 else (y * y).sum())
        n = y.shape[0]
        # d log det / d log s = n: the probed trace of Q^{-1} Q is the number of vertices
        return {"value": np.float64(0.5 * S * t.sum() - 0.5 * s * quad),
                "grad": np.array([k2 * (0.5 * S * dk.sum() - 0.5 * s * dquad), s * (0.5 * S * n / s - 0.5 * quad)])}
    if f == "batch":
        if sum(s * s for _, s in _batch_shapes(case)) > 9e6:
            return None
        logdet, grad, stored = [], [], {}
        for (p, s), k in zip(_batch_shapes(case), _batch_kappa2(case, seed)):
            t, sd, _ = _closed(p, (s, s), False, 4 if p == 5 else 2, float(k),
                               colour=stored.setdefault((p, s), _lattice_colours(p, (s, s), False, 4 if p == 5 else 2)))
            logdet.append(t.sum())
            grad.append(sd.sum() if p == 5 else np.nan)
        return {"logdet": np.array(logdet), "grad": np.array(grad)}
    if f == "mesh":
        apply, K = _fem(case, seed)
        if K.shape[0] > 1.2e5:
            return None
        t, s, _ = _by_cg(apply, _mesh_colours(K, case["alpha"], case["distance"]))
        return {"logdet": np.float64(t.sum()), "terms": t, "seeds": s}
    dims, k2 = _dims(case), _kappa2(case, seed)
    n = int(np.prod(dims))
    if case["periodic"] and n > 4e5:
        return None
    colour = _lattice_colours(case["points"], dims, case["periodic"], case["distance"])
    ids = [p for p in case["grad"].split(",") if p]
    if not case["field"] and case["tau"] == 0:
        t, s, dk = _closed(case["points"], dims, case["periodic"], case["distance"], k2, colour=colour)
        g = {"kappa2": dk.sum(), "scale": float(n)}
    else:
        field = torch.from_numpy(_field(case, seed)).cuda() if case["field"] else torch.ones((), device="cuda").double()
        mask = torch.from_numpy(_mask(case, seed)).cuda().double() if case["tau"] > 0 else torch.zeros(n, device="cuda").double()
        t, s, own = _by_cg(_lattice_apply(dims, case["periodic"], k2 * field + case["tau"] * mask), colour)
        g = {"kappa2": float((field * own).sum()), "tau": float((mask * own).sum()), "scale": float(n)}
    if ids:
        return {"logdet": np.float64(t.sum()), "grad": np.array([g[p] for p in ids])}
    return {"logdet": np.float64(t.sum()), "terms": t, "seeds": s}
