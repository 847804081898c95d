"""Edge cases of the method through the C ABI, against the oracle or LAPACK:
one block (c is empty and Fig. 3 is one LU solve), everything dropped (c is
empty, DDPS is block Jacobi inside the Krylov loop), ragged partitions with
one-row blocks, a tiny system, the identity, and batches that mix these."""

import ctypes

import numpy as np
import pytest
import scipy.sparse as sp

import workloads as W
from gpu_helpers import dev, host, make_solver, relerr
from oracle.ddps_oracle import DDPSOracle
from paper_1008_1700_gb300 import Solver, native as N

pytestmark = pytest.mark.gpu

FP64 = dict(factor_prec=N.DDPS_FP64, spike_prec=N.DDPS_FP64, ghat_prec=N.DDPS_FP64,
            inner_prec=N.DDPS_FP64)
MIXED_TC = dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3, ghat_prec=N.DDPS_FP16,
                inner_prec=N.DDPS_FP32, update_prec=N.DDPS_BF16X3)


def _problem(A, block_ptr, seed=0):
    A = sp.csr_matrix(A)
    A.sort_indices()
    x = np.random.default_rng(seed).uniform(-1, 1, A.shape[0])
    return W.Problem(n=A.shape[0], rowptr=A.indptr.astype(np.int32),
                     colind=A.indices.astype(np.int32), values=A.data.astype(np.float64),
                     block_ptr=np.asarray(block_ptr, dtype=np.int64), f=A @ x, x_true=x)


def _check_solve(P, opts, drop=None, tol=1e-12, max_outer=None):
    S = make_solver(P, drop, tol_out=tol, tol_in=1e-8, maxit_in=300, **opts)
    x, info = S.solve(dev(P.f))
    assert info["status"] == "DDPS_OK", info
    x = host(x)
    A = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr, spikes=False).A
    assert np.max(np.abs(P.f - A @ x)) / np.max(np.abs(P.f)) <= tol
    assert relerr(x, np.linalg.solve(A.toarray(), P.f)) <= 1e-8
    if max_outer is not None:
        assert info["outer_iterations"] <= max_outer
    return S, info


@pytest.mark.parametrize("opts", [FP64, MIXED_TC], ids=["fp64", "mixed"])
def test_single_block_is_one_lu_solve(opts):
    """p = 1: R = 0, c is empty; the preconditioner is the (FP64) LU solve, so
    FP64 converges at the first half step; reduced calls accept m = 0."""
    P = W.small_random_band(800, 1, 60, seed=5)
    S, info = _check_solve(P, opts, max_outer=0.5 if opts is FP64 else 3.0)
    assert S.m == 0 and info["inner_iterations"] == 0
    assert S.sizes["ghat_entries"] == 0
    S.close()


def test_everything_dropped_is_block_jacobi():
    """A drop threshold above every entry of R: c is empty, P = D~, and the
    outer Krylov iteration alone couples the blocks."""
    P = W.small_random_band(1500, 6, 100, seed=6)
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr, drop=("abs", 1e9))
    assert o.m == 0
    S, info = _check_solve(P, FP64, drop=("abs", 1e9))
    assert S.m == 0 and info["outer_iterations"] > 1.0
    xo, oinfo = o.solve(P.f, tol=1e-12)
    assert abs(info["outer_iterations"] - oinfo["iterations"]) <= 1.0
    S.close()


@pytest.mark.parametrize("opts", [FP64, MIXED_TC], ids=["fp64", "mixed"])
def test_ragged_blocks_with_one_row_blocks(opts):
    """Blocks of 1, 2, 37, 1, 150 and 9 rows of a random diagonally dominant
    matrix: G^ element by element and the solve."""
    P = W.small_random_dd(200, 1, k_off=4, dd=1.5, seed=7)
    P.block_ptr = np.array([0, 1, 3, 40, 41, 191, 200], dtype=np.int64)
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr)
    S = make_solver(P, **opts)
    assert np.array_equal(S.interface(), o.c)
    bound = 1e-11 if opts is FP64 else 6e-4
    for b, ob in enumerate(o.blk):
        q0, q1, cols = S.ghat_layout(b)
        if (q1 - q0) * len(cols):
            scale = max(np.max(np.abs(ob["Ghat"])), 1e-300)
            assert np.max(np.abs(S.ghat_block(b) - ob["Ghat"])) <= bound * scale, b
    S.close()
    _check_solve(P, opts)


def test_tiny_and_identity_systems():
    """n = 2 with two one-row blocks (c = both rows), and A = I in 3 blocks
    (no coupling: x = f at once)."""
    A2 = np.array([[4.0, -1.0], [-2.0, 5.0]])
    _check_solve(_problem(A2, [0, 1, 2]), FP64, max_outer=0.5)
    I = sp.identity(50, format="csr")
    S, info = _check_solve(_problem(I, [0, 20, 21, 50], seed=2), FP64, max_outer=0.5)
    assert S.m == 0
    S.close()


def test_batch_mixing_degenerate_systems():
    """One handle with a single-block system, a system with one-row blocks and
    a slab system, and a zero right-hand side for one of them."""
    probs = [W.small_random_band(300, 1, 30, seed=8),
             W.small_convdiff_2d(10, 10),
             W.small_convdiff_3d(8, [2, 3, 3])]
    S = Solver.from_systems([(p.rowptr, p.colind, p.values, p.block_ptr) for p in probs],
                            tol_out=1e-12, tol_in=1e-8, **FP64)
    S.factor(dev(S.values_host))
    fs = [p.f.copy() for p in probs]
    fs[1][:] = 0.0
    x, info = S.solve(dev(np.concatenate(fs)))
    assert info["status"] == "DDPS_OK"
    x = host(x)
    for k, p in enumerate(probs):
        xk = x[S.sys_row_ptr[k]:S.sys_row_ptr[k + 1]]
        A = DDPSOracle(p.n, p.rowptr, p.colind, p.values, p.block_ptr, spikes=False).A
        if k == 1:
            assert np.all(xk == 0.0)
        else:
            assert relerr(xk, np.linalg.solve(A.toarray(), fs[k])) <= 1e-9, k
    S.close()


def test_direct_chain_with_a_one_sided_coupling():
    """A chain where column dropping removes the coupling of one block to its
    predecessor (an S_b with no correction): the direct reduced solve still
    solves G^ exactly (to FP32)."""
    P = W.small_convdiff_3d(10, [3, 4, 3], b=(0.0, 0.0, 40.0))
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr, drop=("column", 0.5))
    S = make_solver(P, ("column", 0.5), reduced_solver=N.DDPS_REDUCED_DIRECT, **FP64)
    g = np.random.default_rng(3).standard_normal(o.m)
    zo, _ = o.reduced_solve(g, mode="direct")
    assert relerr(host(S.reduced_solve(dev(g))), zo) <= 1e-4
    S.close()


@pytest.mark.parametrize("name,N_,p,form", [
    ("one_cta", 12, 3, "half"),          # a single CTA holds the system
    ("held", 64, 4, "half"),             # a cluster, rows split unevenly
    ("held_float", 90, 7, "float"),      # odd sizes, ragged row groups and vectors
    ("held_double", 40, 3, "double"),    # FP64 sums and scalars
    ("held_limit", 160, 8, "half"),      # near the largest that shared memory holds
    ("streamed", 200, 10, "half"),       # a cluster, rows of G^ streamed
    ("loop", 256, 16, "half"),           # beyond a cluster: the launch-per-step loop
])
def test_reduced_solve_paths(name, N_, p, form):
    """The reduced solve meets tol_in on the stored G^ for every size class.  The residual
    is formed in FP64 from the stored blocks; rounding z^ to FP32 adds about 1e-7 to
    the 1e-5 that the iteration stops at, so 1.1e-5 bounds it."""
    opts = {"half": dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3, ghat_prec=N.DDPS_FP16,
                         inner_prec=N.DDPS_FP32),
            "float": dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_FP32, ghat_prec=N.DDPS_FP32,
                          inner_prec=N.DDPS_FP64),
            "double": FP64}[form]
    P = W.small_convdiff_2d(N_, p, seed=N_)
    S = make_solver(P, tol_in=1e-5, maxit_in=300, **opts)
    rng = np.random.default_rng(N_)
    for scale in (1.0, 1e-25, 0.0):  # the scaled copy: squares below FP32's range
        g = scale * rng.uniform(-1, 1, S.m)
        z = host(S.reduced_solve(dev(g)))
        r = g - z
        for b in range(p):
            q0, q1, cols = S.ghat_layout(b)
            r[q0:q1] -= S.ghat_block(b) @ z[cols]
        assert np.linalg.norm(r) <= 1.1e-5 * np.linalg.norm(g), (name, scale)


@pytest.mark.parametrize("autotune", [0, 1])
@pytest.mark.parametrize("rows", [1004, 1024, 2048])
def test_block_solve_front_at_48_kb(rows, autotune):
    """Dense fronts whose sweeps take just under 48 KB of dynamic shared memory (static bytes
    of the kernel beside it)."""
    rng = np.random.default_rng(rows)
    n = rows + 4
    A = np.zeros((n, n))
    A[:rows, :rows] = rng.uniform(-1.0, 1.0, (rows, rows))
    A[0, rows] = A[rows, 0] = 1.0
    A[np.arange(n), np.arange(n)] = 2.0 * rows
    M = sp.csr_matrix(A)
    S = Solver(M.indptr, M.indices, np.array([0, rows, n]), factor_prec=N.DDPS_FP64,
               spike_prec=N.DDPS_FP64, ghat_prec=N.DDPS_FP64, inner_prec=N.DDPS_FP64,
               autotune=autotune)
    S.factor(dev(M.data))
    x, _ = S.solve(dev(A @ np.ones(n)))
    # dominance 2: condition below 3, |x - 1| <= 3 (n + rounding of the right-hand side) eps
    assert np.max(np.abs(host(x) - 1.0)) <= 3 * 2 * n * 2.0 ** -53 + 1e-12


@pytest.mark.parametrize("rows", [256, 257, 384, 515, 641, 1301])
def test_fp32_wide_front_inverses(rows):
    """Block solves through one dense FP32 front: its triangular inverses come from doubling
    steps of 128, 256, .. pivots with ragged last blocks and any row stride."""
    rng = np.random.default_rng(rows)
    n = rows + 3
    A = np.zeros((n, n))
    A[:rows, :rows] = rng.uniform(-1.0, 1.0, (rows, rows))
    A[0, rows] = A[rows, 0] = 1.0
    A[np.arange(n), np.arange(n)] = 0.0
    A[np.arange(n), np.arange(n)] = 1.5 * np.abs(A).sum(axis=1) + 0.1
    M = sp.csr_matrix(A)
    S = Solver(M.indptr, M.indices, np.array([0, rows, n]), factor_prec=N.DDPS_FP32,
               spike_prec=N.DDPS_FP32, ghat_prec=N.DDPS_FP32, inner_prec=N.DDPS_FP32)
    S.factor(dev(M.data))
    y = rng.uniform(-1.0, 1.0, n)
    x = host(S.block_solve(dev(y)))[:rows]
    r = A[:rows, :rows] @ x - y[:rows]
    # dominance: |L||U| <= 3 |M|; rows roundings each for the factors, the inverses and the
    # two triangular products of the solve
    assert np.linalg.norm(r) <= 3 * 4 * rows * 2.0 ** -24 * np.linalg.norm(np.abs(A[:rows, :rows]) @ np.abs(x))
    S.close()


@pytest.mark.parametrize("prec", [N.DDPS_FP32, N.DDPS_FP64])
@pytest.mark.parametrize("rows", [1, 3, 8, 9, 31, 32, 33, 64, 65, 90, 96, 97, 127, 128])
def test_dense_front_edges(rows, prec):
    """Block solves through one dense front at the edges of the register rows, the pivot
    panels and the four-column groups of the inverses."""
    rng = np.random.default_rng(rows)
    n = rows + 3
    A = np.zeros((n, n))
    A[:rows, :rows] = rng.uniform(-1.0, 1.0, (rows, rows))
    A[0, rows] = A[rows, 0] = 1.0
    A[np.arange(n), np.arange(n)] = 0.0
    A[np.arange(n), np.arange(n)] = 1.5 * np.abs(A).sum(axis=1) + 0.1
    M = sp.csr_matrix(A)
    S = Solver(M.indptr, M.indices, np.array([0, rows, n]), factor_prec=prec, spike_prec=prec,
               ghat_prec=prec, inner_prec=prec)
    S.factor(dev(M.data))
    y = rng.uniform(-1.0, 1.0, n)
    x = host(S.block_solve(dev(y)))[:rows]
    D = A[:rows, :rows]
    u = 2.0 ** (-24 if prec == N.DDPS_FP32 else -53)
    # dominance: |L||U| <= 3 |D|; rows (and a conversion's) roundings each for the factors,
    # the inverses and the two triangular products
    assert np.linalg.norm(D @ x - y[:rows]) <= 3 * 4 * (rows + 1) * u * np.linalg.norm(np.abs(D) @ np.abs(x))
    S.close()


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_statistics_of_a_batch_with_an_uncoupled_system(form):
    """A system without coupling columns takes no part in the reduced solve: the counts
    returned are those of the coupled one alone, whatever the device memory held before."""
    opts = dict(FP64 if form == "fp64" else MIXED_TC, tol_out=1e-10, tol_in=1e-6)
    a, b = W.small_random_band(300, 1, 30, seed=8), W.small_convdiff_2d(10, 10)

    def run(probs):
        S = Solver.from_systems([(p.rowptr, p.colind, p.values, p.block_ptr) for p in probs], **opts)
        S.factor(dev(S.values_host))
        g = dev(np.linspace(1.0, 2.0, S.m))
        z = host(S.reduced_solve(g))
        info = S.solve(dev(np.concatenate([p.f for p in probs])))[1]
        S.close()
        return z, info
    z1, alone = run([b])
    # every other one of many small blocks full of bytes 0x41 is given back: the next handle's
    # small allocations come from these (memory of a wholly free region is cleared)
    rt = ctypes.CDLL("libcudart.so")
    junk = [ctypes.c_void_p() for _ in range(20000)]
    for q in junk:
        assert rt.cudaMalloc(ctypes.byref(q), ctypes.c_size_t(512)) == 0
        assert rt.cudaMemset(q, 0x41, ctypes.c_size_t(512)) == 0
    for q in junk[::2]:
        assert rt.cudaFree(q) == 0
    z2, both = run([a, b])
    for q in junk[1::2]:
        assert rt.cudaFree(q) == 0
    assert alone["guess_used"] == both["guess_used"] == 0
    assert both["first_inner_iters"] == alone["first_inner_iters"]
    # the uncoupled system may add outer iterations, in which the coupled one takes none
    assert both["inner_iterations"] == alone["inner_iterations"]
    assert np.array_equal(z1, z2)


@pytest.mark.parametrize("ghat", ["FP16", "BF16", "FP32", "FP64"])
@pytest.mark.parametrize("inner", ["FP32", "FP64"])
def test_small_system_inner_iteration_forms_and_guess(ghat, inner):
    """The inner iteration in one launch for every storage of G^ and precision of the vectors:
    the residual on the stored G^ (as in test_reduced_solve_paths), and a guess of the first
    preconditioner application -- a bad one is not used, the answer saves its iterations."""
    if (ghat, inner) == ("FP64", "FP32"):
        pytest.skip("an FP64 G^ needs FP64 vectors")
    fact = dict(factor_prec=N.DDPS_FP64, spike_prec=N.DDPS_FP64) if ghat == "FP64" else \
        dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3)
    P = W.small_convdiff_2d(40, 3, seed=2)
    S = make_solver(P, tol_in=1e-5, maxit_in=300, tol_out=1e-10, **fact,
                    ghat_prec=getattr(N, "DDPS_" + ghat), inner_prec=getattr(N, "DDPS_" + inner))
    g = np.random.default_rng(9).uniform(-1, 1, S.m)
    z = host(S.reduced_solve(dev(g)))
    r = g - z
    for b in range(3):
        q0, q1, cols = S.ghat_layout(b)
        r[q0:q1] -= S.ghat_block(b) @ z[cols]
    assert np.linalg.norm(r) <= 1.1e-5 * np.linalg.norm(g)
    f = dev(P.f)
    _, cold = S.solve(f)
    zhat, _ = S.reduced_solution()
    S.set_reduced_guess(dev(1e3 * np.random.default_rng(3).standard_normal(S.m)))
    x, bad = S.solve(f)
    assert bad["guess_used"] == 0 and bad["first_inner_iters"] == cold["first_inner_iters"]
    S.set_reduced_guess(zhat)
    y, warm = S.solve(f)
    assert warm["status"] == "DDPS_OK" and warm["guess_used"] == 1
    # the guess meets the tolerance but for its own last rounding
    assert warm["first_inner_iters"] <= 1.0 < cold["first_inner_iters"]
    assert relerr(host(y), host(x)) <= 1e-7
    S.close()
