"""ILU(0) block factors (factor_kind ILU0; Sec. 3: the block factors of
Fig. 2 step 2 may be approximate) through the C ABI against the oracle's
ILU(0) (``DDPSOracle(factor="ilu0")``): block solves with L~ U~, the spikes
G^ element by element, and the whole solve, whose outer iteration still
reaches the solution of A x = f."""

import numpy as np
import pytest
import scipy.sparse as sp

import workloads as W
from gpu_helpers import dev, host, make_solver, relerr
from oracle.ddps_oracle import DDPSOracle
from paper_1008_1700_gb300 import Solver, native as N

pytestmark = pytest.mark.gpu

ILU64 = dict(factor_prec=N.DDPS_FP64, spike_prec=N.DDPS_FP64, ghat_prec=N.DDPS_FP64,
             inner_prec=N.DDPS_FP64, factor_kind=N.DDPS_FACTOR_ILU0)
ILU32 = dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_FP32, ghat_prec=N.DDPS_FP32,
             inner_prec=N.DDPS_FP32, factor_kind=N.DDPS_FACTOR_ILU0)

PROBLEMS = {
    "cd2d_24_p3": (lambda: W.small_convdiff_2d(24, 3), None),
    "cd3d_12_slabs": (lambda: W.small_convdiff_3d(12, [3, 5, 4]), None),
    "randdd_301_p7": (lambda: W.small_random_dd(301, 7, seed=9), None),
    "band_3000_abs": (lambda: W.small_random_band(3000, 5, 200, seed=2), ("abs", 1e-4)),
}


@pytest.fixture(scope="module", params=sorted(PROBLEMS))
def case(request):
    make, drop = PROBLEMS[request.param]
    P = make()
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr, drop=drop, factor="ilu0")
    return request.param, P, drop, o


@pytest.mark.parametrize("form,bound", [("fp64", 1e-12), ("fp32", 2e-5)])
def test_ilu_block_solve_and_spikes(case, form, bound):
    name, P, drop, o = case
    S = make_solver(P, drop, **(ILU64 if form == "fp64" else ILU32))
    y = np.random.default_rng(1).standard_normal(P.n)
    assert relerr(host(S.block_solve(dev(y))), o.block_solve(y)) <= bound, name
    assert np.array_equal(S.interface(), o.c)
    for b, ob in enumerate(o.blk):
        q0, q1, cols = S.ghat_layout(b)
        if (q1 - q0) * len(cols) == 0:
            continue
        scale = max(np.max(np.abs(ob["Ghat"])), 1e-300)
        assert np.max(np.abs(S.ghat_block(b) - ob["Ghat"])) <= 10 * bound * scale, (name, b)
    S.close()


@pytest.mark.parametrize("form", ["fp64", "fp32", "fp32_direct"])
def test_ilu_full_solve(case, form):
    name, P, drop, o = case
    opts = dict(ILU64 if form == "fp64" else ILU32)
    if form == "fp32_direct":
        if name.startswith(("randdd", "band")):
            pytest.skip("not a chain of blocks")
        opts["reduced_solver"] = N.DDPS_REDUCED_DIRECT
    S = make_solver(P, drop, tol_out=1e-12, tol_in=1e-6, maxit_in=200, **opts)
    x, info = S.solve(dev(P.f))
    assert info["status"] == "DDPS_OK", info
    x = host(x)
    assert np.max(np.abs(P.f - o.A @ x)) / np.max(np.abs(P.f)) <= 1e-12
    xo = np.linalg.solve(o.A.toarray(), P.f)
    assert relerr(x, xo) <= 1e-8, name
    S.close()


def test_ilu_outer_iterations_against_the_oracle():
    """Same approximate preconditioner on both sides: the outer iteration
    counts of the FP64 GPU solve and of the oracle agree to one step."""
    P = W.small_convdiff_3d(12, [3, 5, 4])
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr, factor="ilu0")
    S = make_solver(P, tol_out=1e-12, tol_in=1e-8, maxit_in=200, **ILU64)
    _, info = S.solve(dev(P.f))
    _, oinfo = o.solve(P.f, tol=1e-12, eps_in=1e-8, maxit_in=200)
    assert info["outer_iterations"] > 1.0
    assert abs(info["outer_iterations"] - oinfo["iterations"]) <= 1.0


def test_ilu_rejects_a_missing_diagonal():
    P = W.small_convdiff_2d(8, 2)
    keep = np.ones(P.nnz, dtype=bool)
    keep[P.rowptr[5]:P.rowptr[6]] = np.arange(P.rowptr[5], P.rowptr[6]) != \
        P.rowptr[5] + int(np.nonzero(P.colind[P.rowptr[5]:P.rowptr[6]] == 5)[0][0])
    colind = P.colind[keep]
    counts = np.diff(P.rowptr) - np.add.reduceat(~keep, P.rowptr[:-1].astype(np.int64))
    rowptr = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    with pytest.raises(N.DDPSError, match="INVALID_ARG.*diagonal"):
        Solver(rowptr, colind, P.block_ptr, **ILU64)


@pytest.mark.parametrize("name,make", [
    ("vector_beyond_shared_memory", lambda: W.small_convdiff_2d(180, 1)),  # 32,400 FP64 rows a block
    ("levels_beyond_the_threads", lambda: W.small_random_dd(6001, 3, k_off=1, seed=4)),
    ("single_rows", lambda: W.small_random_dd(9, 9, k_off=2, seed=5)),      # blocks of one row
])
def test_ilu_one_launch_solves(name, make):
    """The one-launch block solve where its shapes change; FP64 triangular solves in
    the oracle's entry order agree to rounding (the bound of the small cases)."""
    P = make()
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr, factor="ilu0")
    y = np.random.default_rng(3).standard_normal(P.n)
    S = make_solver(P, **ILU64)
    assert relerr(host(S.block_solve(dev(y))), o.block_solve(y)) <= 1e-12
    S.close()


def _launches(S, y):
    n0 = S.launch_count()
    g = host(S.block_solve(dev(y)))
    return g, S.launch_count() - n0


@pytest.mark.parametrize("prec,bound", [(N.DDPS_FP64, 1e-12), (N.DDPS_FP32, 2e-5)])
@pytest.mark.parametrize("n,p,one", [(60000, 2, False), (60000, 100, True)])
def test_ilu_block_solve_route_by_the_width_of_the_levels(n, p, one, prec, bound):
    """Few levels of thousands of rows in two blocks take a launch per level, which spreads
    their rows over the GPU; the same levels in many blocks take one launch.  The blocks are
    lower triangular, so ILU(0) is exact."""
    rng = np.random.default_rng(p)
    bs, levels = n // p, 8
    row = np.repeat(np.arange(n), 3)
    level = row % bs * levels // bs
    row, level = row[level > 0], level[level > 0]
    col = row - row % bs + (level - 1) * bs // levels + rng.integers(0, bs // levels - 1, len(row))
    A = sp.csr_matrix((rng.uniform(-0.3, 0.3, len(row)), (row, col)), shape=(n, n))
    A = A + 2.0 * sp.identity(n)
    A = A + sp.csr_matrix(([0.1], ([0], [n - 1])), shape=(n, n))  # blocks coupled by one entry
    A = sp.csr_matrix(A)
    A.sort_indices()
    S = Solver(A.indptr, A.indices, np.arange(p + 1) * bs, **dict(ILU64 if prec == N.DDPS_FP64 else ILU32))
    S.factor(dev(A.data))
    y = rng.standard_normal(n)
    g, launches = _launches(S, y)
    D = sp.csr_matrix(sp.tril(A))
    assert relerr(D @ g, y) <= bound
    assert (launches == 1) == one, launches
    S.close()


def test_ilu_block_solve_of_an_arrow():
    """A row and a column of full width in every block: rows are not padded to the widest, the
    sweeps take a launch per level."""
    n, p = 600, 2
    rng = np.random.default_rng(2)
    A = sp.lil_matrix(sp.diags([rng.uniform(-1, 1, n - 1), np.full(n, 500.0), rng.uniform(-1, 1, n - 1)],
                               [-1, 0, 1]))
    for b in range(p):
        r0, r1 = b * n // p, (b + 1) * n // p
        A[r1 - 1, r0:r1 - 1] = rng.uniform(-1, 1, r1 - r0 - 1)
        A[r0:r1 - 1, r1 - 1] = rng.uniform(-1, 1, (r1 - r0 - 1, 1))
    A = sp.csr_matrix(A)
    A.sort_indices()
    cuts = np.arange(p + 1, dtype=np.int64) * (n // p)
    o = DDPSOracle(n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, cuts, factor="ilu0")
    y = rng.standard_normal(n)
    for opts, bound in ((ILU64, 1e-12), (ILU32, 2e-5)):
        S = Solver(A.indptr, A.indices, cuts, **opts)
        S.factor(dev(A.data))
        g, launches = _launches(S, y)
        assert relerr(g, o.block_solve(y)) <= bound
        assert launches > 100
        S.close()
