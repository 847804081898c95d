"""Performance cases: the work a user of the solver has it do, through the
public ``Solver`` and ``GuessNet`` entry points.

A case is a dict of plain values.  ``kind`` says which calls one pass makes:

* ``solve``: new matrix values on a known pattern, ``Solver.factor`` and then
  ``Solver.solve`` -- one step of a time integration or a Newton loop, where
  the symbolic analysis is kept and the numbers are new;
* ``resolve``: ``Solver.solve`` alone with several right-hand sides against
  factors that are kept;
* ``block_solve``, ``spmv``, ``reduced_matvec``: one component call, as a
  program does that runs its own outer iteration around the solver's parts;
* ``mlp_grad``: loss and gradients of one full-batch training step of the
  network that predicts the reduced system's starting vector;
* ``mlp_predict``: one prediction with it.

Systems are the synthetic families the package is used on: 2-D and 3-D
convection-diffusion on grid-line and slab blocks, batches of uneven 2-D
systems, and nonsymmetric random bands with a few long-range entries.  The
right-hand side is f = A x for a random x, so x is the exact answer.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1008_1700_gb300 import native as N
from paper_1008_1700_gb300.learned import GuessNet
from paper_1008_1700_gb300.solver import Solver

# ---------------------------------------------------------------------------
# option sets
# ---------------------------------------------------------------------------
# The outer tolerance is tight (a residual of 1e-12) so that x is determined
# by the system and not by where the iteration happened to stop.
_BASE = dict(tol_out=1e-12, maxit_out=1000, tol_in=1e-4, maxit_in=100)
_TC = dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3, inner_prec=N.DDPS_FP32,
           update_prec=N.DDPS_BF16X3)
_FORMS = {
    # the defaults: FP64 everywhere
    "fp64": {},
    # FP32 factors, tensor-core spikes, FP16 reduced matrix: the throughput form
    "mixed": dict(_TC, ghat_prec=N.DDPS_FP16),
    # the same with the reduced matrix in FP32 / BF16
    "mixed_g32": dict(_TC, ghat_prec=N.DDPS_FP32),
    "mixed_gbf16": dict(_TC, ghat_prec=N.DDPS_BF16),
    # the reduced system solved directly by block LU
    "direct": dict(_TC, ghat_prec=N.DDPS_FP16, reduced_solver=N.DDPS_REDUCED_DIRECT),
    # the reduced matrix applied by block solves, never stored
    "implicit": dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_FP32, ghat_prec=N.DDPS_FP32,
                     inner_prec=N.DDPS_FP32, ghat_mode=N.DDPS_GHAT_IMPLICIT),
    # ILU(0) block factors
    "ilu": dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_FP32, ghat_prec=N.DDPS_FP16,
                inner_prec=N.DDPS_FP32, factor_kind=N.DDPS_FACTOR_ILU0),
}


def _options(case):
    o = dict(_BASE, **_FORMS[case["form"]])
    if case.get("drop_abs"):
        o.update(drop_mode=N.DDPS_DROP_ABS, drop_tol=case["drop_abs"])
    return o


# ---------------------------------------------------------------------------
# systems: the pattern depends on the case alone (a program analyses it once),
# the values and the solution on the seed
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=512)
def _grid(side, dim):
    """5- or 7-point pattern on a side^dim grid (x fastest): rowptr, colind and
    the stencil position of every entry (0 = diagonal, 1 + 2 a / 2 + 2 a = the
    lower / upper neighbour along axis a)."""
    n = side ** dim
    idx = np.arange(n, dtype=np.int64)
    order = [(a, -1) for a in reversed(range(dim))] + [(0, 0)] + [(a, 1) for a in range(dim)]
    cols = np.empty((n, len(order)), dtype=np.int64)
    ok = np.ones((n, len(order)), dtype=bool)
    code = np.empty(len(order), dtype=np.int8)
    for q, (a, d) in enumerate(order):
        cols[:, q] = idx + d * side ** a
        if d:
            c = idx // side ** a % side + d
            ok[:, q] = (c >= 0) & (c < side)
        code[q] = 0 if d == 0 else (1 + 2 * a if d < 0 else 2 + 2 * a)
    rowptr = np.zeros(n + 1, dtype=np.int32)
    np.cumsum(ok.sum(axis=1), out=rowptr[1:])
    return rowptr, cols[ok].astype(np.int32), np.broadcast_to(code, ok.shape)[ok]


def _grid_values(side, dim, b):
    h = 1.0 / (side + 1)
    t = np.empty(1 + 2 * dim)
    t[0] = 2.0 * dim
    for a in range(dim):
        t[1 + 2 * a] = -1.0 - b[a] * h / 2.0
        t[2 + 2 * a] = -1.0 + b[a] * h / 2.0
    return t[_grid(side, dim)[2]]


@functools.lru_cache(maxsize=512)
def _cuts(side, dim, p):
    """p blocks of whole grid lines (2-D) or planes (3-D), uneven: equal shares
    and then a few seeded moves of one line or plane between blocks."""
    sizes = [side // p + (1 if i < side % p else 0) for i in range(p)]
    rng = np.random.default_rng([side, dim, p])
    for _ in range(p // 4):
        i, j = (int(v) for v in rng.integers(0, p, 2))
        if i != j and sizes[j] >= 3:
            sizes[i] += 1
            sizes[j] -= 1
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64) * side ** (dim - 1)


@functools.lru_cache(maxsize=4)
def _band(n, hw):
    """11 distinct off-diagonal columns per row within +-hw, one in a hundred
    anywhere, and the diagonal; columns sorted."""
    k = 11
    rng = np.random.default_rng([n, hw])

    def pick(rows):
        near = rows[:, None] + rng.integers(-hw, hw + 1, (len(rows), k))
        return np.where(rng.random((len(rows), k)) < 0.01, rng.integers(0, n, near.shape), near)

    rows = np.arange(n, dtype=np.int64)
    cols = np.empty((n, k + 1), dtype=np.int64)
    bad = rows
    while len(bad):
        c = np.concatenate([pick(bad), bad[:, None]], axis=1)
        c.sort(axis=1)
        cols[bad] = c
        wrong = (c[:, 0] < 0) | (c[:, -1] >= n) | (c[:, 1:] == c[:, :-1]).any(axis=1)
        bad = bad[wrong]
    rowptr = (np.arange(n + 1, dtype=np.int64) * (k + 1)).astype(np.int32)
    return rowptr, cols.astype(np.int32).ravel(), (cols == rows[:, None]).ravel()


def _product(rowptr, colind, values, x):
    return np.add.reduceat(values * x[colind], rowptr[:-1].astype(np.int64))


@functools.lru_cache(maxsize=64)
def _sides(count, lo, hi):
    return [int(v) for v in np.random.default_rng([count, lo, hi]).integers(lo, hi + 1, count)]


def _systems(case, seed):
    """[(rowptr, colind, values, block_ptr)] of the case's systems and the
    solution vectors."""
    rng = np.random.default_rng([seed, 11])
    out, xs = [], []
    if case["family"] == "band":
        n = case["n"]
        rowptr, colind, diag = _band(n, case["hw"])
        values = rng.standard_normal(len(colind))
        values[diag] = 0.0
        values[diag] = 1.2 * np.abs(values).reshape(n, -1).sum(axis=1)
        cuts = np.array([i * n // case["p"] for i in range(case["p"] + 1)], dtype=np.int64)
        out.append((rowptr, colind, values, cuts))
    else:
        dim = 3 if case["family"] == "cd3d" else 2
        sides = ([case["side"]] if case["family"] != "batch"
                 else _sides(case["count"], case["side_lo"], case["side_hi"]))
        for side in sides:
            # convection up to 50 per axis, inside the central scheme's limit
            b = rng.uniform(0.0, min(50.0 if dim == 3 else 20.0, 1.6 * (side + 1)), dim)
            rowptr, colind, _ = _grid(side, dim)
            out.append((rowptr, colind, _grid_values(side, dim, b), _cuts(side, dim, case["p"])))
    for s in out:
        xs.append(rng.uniform(-1.0, 1.0, len(s[0]) - 1))
    return out, xs


def _make_solver(case, systems):
    opts = _options(case)
    if case["family"] == "batch":
        return Solver.from_systems(systems, **opts)
    rowptr, colind, values, cuts = systems[0]
    return Solver(rowptr, colind, cuts, values_host=values if case.get("drop_abs") else None,
                  **opts)


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # smallest whole step: a 2-D model problem of 576 unknowns with default options
        dict(name="cd2d_24_p3_fp64", kind="solve", family="cd2d", side=24, p=3, form="fp64"),
        # one small system in the throughput form: latency and launches
        dict(name="cd2d_64_p4_mixed", kind="solve", family="cd2d", side=64, p=4, form="mixed"),
        # the headline: one 3-D step of 262,144 unknowns on 16 uneven slabs
        dict(name="cd3d_64_p16_mixed", kind="solve", family="cd3d", side=64, p=16, form="mixed"),
        # many independent uneven 2-D systems in one handle: parameter studies, ensembles
        dict(name="cd2d_batch256_mixed", kind="solve", family="batch", count=256, side_lo=32,
             side_hi=128, p=8, form="mixed"),
        # the largest: an unstructured band matrix with large fronts and the element-wise drop rule
        dict(name="band_300k_p38_mixed", kind="solve", family="band", n=300_000, hw=2000, p=38,
             drop_abs=1e-4, form="mixed"),
        # the 3-D step with the reduced matrix applied by block solves
        dict(name="cd3d_64_p16_implicit", kind="solve", family="cd3d", side=64, p=16,
             form="implicit"),
        # a 3-D step with default options (FP64 everywhere)
        dict(name="cd3d_48_p8_fp64", kind="solve", family="cd3d", side=48, p=8, form="fp64"),
        # the 3-D step with the direct reduced solver
        dict(name="cd3d_48_p8_direct", kind="solve", family="cd3d", side=48, p=8, form="direct"),
        # new right-hand sides for a matrix that stays
        dict(name="cd3d_48_p8_resolve4", kind="resolve", family="cd3d", side=48, p=8, nrhs=4,
             form="mixed"),
        # approximate block factors, an odd grid on ragged slabs
        dict(name="cd3d_37_p5_ilu", kind="solve", family="cd3d", side=37, p=5, form="ilu"),
        # one block solve of a program with its own outer iteration
        dict(name="cd2d_127_p8_block_solve", kind="block_solve", family="cd2d", side=127, p=8,
             form="fp64"),
        # training of the starting-vector network on 100 steps of the 48^3 sequence
        dict(name="mlp_grad_100x32256", kind="mlp_grad", batch=100, d_in=2, hidden=256, layers=3,
             d_out=32256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["resolve"] * 2 + ["block_solve", "spmv", "reduced_matvec",
                                                         "mlp_grad", "mlp_predict"])
    if kind in ("mlp_grad", "mlp_predict"):
        return dict(kind=kind, batch=_log(rng, 8, 200) if kind == "mlp_grad" else rng.choice([1, 1, 4]),
                    d_in=rng.choice([1, 2]), hidden=256, layers=3, d_out=_log(rng, 300, 40000))
    if kind in ("block_solve", "spmv", "reduced_matvec"):
        family, forms = rng.choice(["cd2d", "cd3d"]), ["fp64"]
    else:
        family = rng.choice(["cd2d", "cd2d", "cd3d", "cd3d", "batch", "band"])
        forms = (["mixed", "mixed", "mixed_g32", "mixed_gbf16"] if family == "band" else
                 ["mixed", "mixed", "mixed_g32", "mixed_gbf16", "implicit", "fp64", "direct", "ilu"])
    form = rng.choice(forms)
    case = dict(kind=kind, family=family, form=form)
    if family == "cd2d":
        case["side"] = _log(rng, 16, 72 if form == "ilu" else 256)
        case["p"] = rng.randint(2, min(16, case["side"] // 4))
    elif family == "cd3d":
        case["side"] = _log(rng, 12, 34 if form == "ilu" else 40 if form in ("fp64", "direct") else 64)
        case["p"] = rng.randint(2, max(2, case["side"] // 4))
        if case["side"] // case["p"] > 6:  # slabs as thin as the method is used with
            case["p"] = case["side"] // 6 + 1
    elif family == "batch":
        case["side_lo"] = rng.randint(16, 40)
        case["side_hi"] = case["side_lo"] + rng.randint(0, 60)
        case["count"] = _log(rng, 3, 24 if form in ("fp64", "ilu") else 200)
        case["p"] = rng.randint(2, 4 if form == "ilu" else 8)
    else:
        case["n"] = _log(rng, 4000, 250_000)
        case["p"] = max(2, case["n"] // _log(rng, 2000, 8000))
        case["hw"] = _log(rng, 50, min(2000, case["n"] // case["p"] // 2))
        case["drop_abs"] = rng.choice([0.0, 1e-4])
    if kind == "resolve":
        case["nrhs"] = rng.randint(1, 4)
    return case


# ---------------------------------------------------------------------------
# one case
# ---------------------------------------------------------------------------
def _mlp_arrays(case, seed):
    """Inputs (normalised coefficients of consecutive steps) and targets (smooth
    in them, scaled to 1) of the network, float32."""
    rng = np.random.default_rng([seed, 5])
    t = np.arange(case["batch"]) + rng.uniform(0, 200)
    X = np.stack([np.sin(2 * np.pi * t / 200), np.cos(2 * np.pi * t / 200)], axis=1)[:, :case["d_in"]]
    T = np.sin(X[:, :1] * 3 + rng.uniform(0, 6, case["d_out"])[None, :]) * rng.uniform(0, 1, case["d_out"])
    return X.astype(np.float32), T.astype(np.float32)


def _mlp_params(case, seed):
    """Weights as after a short training (He-scaled, a small last layer, small
    biases) in the library's flat order, float32."""
    rng = np.random.default_rng([seed, 7])
    dims = [case["d_in"]] + [case["hidden"]] * case["layers"] + [case["d_out"]]
    parts = []
    for l, (a, b) in enumerate(zip(dims, dims[1:])):
        bound = math.sqrt(6.0 / a) * (0.1 if l == len(dims) - 2 else 1.0)
        parts += [rng.uniform(-bound, bound, a * b), rng.uniform(-0.05, 0.05, b)]
    return dims, np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    st = {"case": case}
    if case["kind"].startswith("mlp"):
        X, T = _mlp_arrays(case, seed)
        st["net"] = GuessNet(case["d_in"], case["d_out"], case["hidden"], case["layers"])
        st["net"].params.copy_(torch.from_numpy(_mlp_params(case, seed)[1]))
        st["X"], st["T"] = torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")
        return st
    systems, xs = _systems(case, seed)
    S = st["S"] = _make_solver(case, systems)
    st["values"] = torch.tensor(np.concatenate([s[2] for s in systems]), device="cuda")
    kind = case["kind"]
    if kind == "solve":
        f = np.concatenate([_product(s[0], s[1], s[2], x) for s, x in zip(systems, xs)])
        st["f"] = torch.tensor(f, device="cuda")
        return st
    S.factor(st["values"])
    if kind == "resolve":
        f = [np.concatenate([_product(s[0], s[1], s[2], x) for s, x in zip(systems, X)])
             for X in _solutions(case, seed, xs)]
        st["f"] = torch.tensor(np.stack(f), device="cuda")
    else:
        st["y"] = torch.tensor(_vector(seed, S.m if kind == "reduced_matvec" else S.n), device="cuda")
    return st


def _solutions(case, seed, xs):
    rng = np.random.default_rng([seed, 13])
    return [xs] + [[rng.uniform(-1.0, 1.0, len(x)) for x in xs] for _ in range(case["nrhs"] - 1)]


def _vector(seed, n):
    return np.random.default_rng([seed, 17]).uniform(-1.0, 1.0, n)


def run(state):
    kind = state["case"]["kind"]
    if kind == "mlp_grad":
        grads, loss = state["net"].backward(state["X"], state["T"])
        return {"grads": grads, "loss": loss}
    if kind == "mlp_predict":
        return state["net"].forward(state["X"])
    S = state["S"]
    if kind == "solve":
        S.factor(state["values"])
        return S.solve(state["f"])[0]
    if kind == "resolve":
        return S.solve(state["f"])[0]
    return getattr(S, kind)(state["y"])


@functools.lru_cache(maxsize=64)
def _sizes(key):
    case = dict(key)
    systems, _ = _systems(case, 0)
    if case["family"] == "batch":
        from paper_1008_1700_gb300.solver import stack_systems
        rowptr, colind, values, cuts, sbp, _ = stack_systems(systems)
    else:
        (rowptr, colind, values, cuts), sbp = systems[0], None
    return N.ddps_symbolic(rowptr, colind, cuts, sbp, values,
                           N.default_options(**_options(case)))[0]


def work(case):
    kind = case["kind"]
    if kind.startswith("mlp"):
        dims = [case["d_in"]] + [case["hidden"]] * case["layers"] + [case["d_out"]]
        par = sum(a * b + b for a, b in zip(dims, dims[1:]))
        mac = sum(a * b for a, b in zip(dims, dims[1:]))
        io = case["batch"] * (dims[0] + dims[-1])
        if kind == "mlp_predict":
            return {"bytes": 4 * (par + io), "flops": 2 * case["batch"] * mac}
        # parameters and targets in, gradients out; the first layer has no input gradient
        return {"bytes": 4 * (2 * par + io),
                "flops": 2 * case["batch"] * (3 * mac - dims[0] * dims[1])}
    s = _sizes(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    n, nnz, form = s["n"], s["nnz"], case["form"]
    matrix = 12 * nnz + 4 * (n + 1)
    fs = 8 if form == "fp64" else 4
    gs = {"fp64": 8, "mixed_g32": 4}.get(form, 2)
    stored = 0 if form == "implicit" else s["ghat_entries"] * gs
    factors = s["factor_lu_entries"] * fs
    if kind == "spmv":
        return {"bytes": matrix + 16 * n, "flops": 2 * nnz}
    if kind == "block_solve":
        return {"bytes": factors + 16 * n, "flops": 2 * s["factor_lu_entries"]}
    if kind == "reduced_matvec":
        return {"bytes": stored + 16 * s["m"], "flops": 2 * s["ghat_entries"]}
    if kind == "resolve":  # the kept factors and the matrix, read once; f in and x out
        return {"bytes": matrix + factors + stored + 16 * n * case["nrhs"],
                "flops": 2 * case["nrhs"] * (nnz + s["factor_lu_entries"])}
    # the matrix and f in, x out; the block factorisation and one residual
    return {"bytes": matrix + 16 * n, "flops": s["factor_flops"] + 2 * nnz}


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("mlp"):
        return _mlp_exact(case, seed)
    systems, xs = _systems(case, seed)
    if kind == "solve":
        return np.concatenate(xs)
    if kind == "resolve":
        return np.stack([np.concatenate(X) for X in _solutions(case, seed, xs)])
    if kind == "reduced_matvec":
        return None
    rowptr, colind, values, cuts = systems[0]
    y = _vector(seed, len(rowptr) - 1)
    if kind == "spmv":
        return _product(rowptr, colind, values, y)
    if max(np.diff(cuts)) > 4096:
        return None
    out = np.empty_like(y)
    for r0, r1 in zip(cuts[:-1], cuts[1:]):
        e = slice(rowptr[r0], rowptr[r1])
        rows = np.repeat(np.arange(r1 - r0), np.diff(rowptr[r0:r1 + 1]))
        keep = (colind[e] >= r0) & (colind[e] < r1)
        D = np.zeros((r1 - r0, r1 - r0))
        D[rows[keep], colind[e][keep] - r0] = values[e][keep]
        out[r0:r1] = np.linalg.solve(D, y[r0:r1])
    return out


def _mlp_exact(case, seed):
    X, T = (torch.tensor(a, dtype=torch.float64) for a in _mlp_arrays(case, seed))
    dims, params = _mlp_params(case, seed)
    p, o, leaves = torch.from_numpy(params).double(), 0, []
    A = X
    for l, (a, b) in enumerate(zip(dims, dims[1:])):
        W = p[o:o + a * b].reshape(b, a).clone().requires_grad_()
        c = p[o + a * b:o + a * b + b].clone().requires_grad_()
        o += a * b + b
        leaves += [W, c]
        A = A @ W.T + c
        if l < len(dims) - 2:
            A = torch.relu(A)
    if case["kind"] == "mlp_predict":
        return A.detach()
    loss = 0.5 / case["batch"] * ((A - T) ** 2).sum()
    loss.backward()
    return {"grads": torch.cat([v.grad.reshape(-1) for v in leaves]),
            "loss": loss.detach().reshape(1)}
