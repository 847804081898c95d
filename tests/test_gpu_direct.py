"""Direct solve of the reduced system (Fig. 3 step 6.3 "directly"; Sec. 3
direct mode) for chains of blocks, through the C ABI, against the oracle's
dense solve of the same G^ (``DDPSOracle.reduced_solve(mode="direct")``) and
against the oracle's whole solve.  The block LU of G^ runs in FP32, so a
reduced solve matches to FP32 accuracy; the FP64 outer iteration then
recovers the full solution, with no inner iterations."""

import numpy as np
import pytest

import workloads as W
from gpu_helpers import dev, host, make_solver, relerr
from oracle.ddps_oracle import DDPSOracle
from paper_1008_1700_gb300 import Solver, native as N

pytestmark = pytest.mark.gpu

FP64_DIRECT = dict(factor_prec=N.DDPS_FP64, spike_prec=N.DDPS_FP64, ghat_prec=N.DDPS_FP64,
                   inner_prec=N.DDPS_FP64, reduced_solver=N.DDPS_REDUCED_DIRECT)
# the benched mixed form (FP32 factors, tensor-core spikes and LU updates, FP16 G^)
MIXED_DIRECT = dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3, ghat_prec=N.DDPS_FP16,
                    inner_prec=N.DDPS_FP32, update_prec=N.DDPS_BF16X3,
                    reduced_solver=N.DDPS_REDUCED_DIRECT)

CHAINS = {
    "cd2d_24_p3": lambda: W.small_convdiff_2d(24, 3),
    "cd2d_cfg1": lambda: W.cfg1(),
    "cd3d_12_slabs": lambda: W.small_convdiff_3d(12, [3, 5, 4]),
    # 45 x 45 planes (2,025 rows per interface: 32 Gauss-Jordan steps, the last one
    # 41 columns wide, and ragged 128 x 128 GEMM tiles)
    "cd3d_45_slabs9": lambda: W.small_convdiff_3d(45, [5] * 9),
}


@pytest.fixture(scope="module", params=sorted(CHAINS))
def chain(request):
    P = CHAINS[request.param]()
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr,
                   spikes=request.param != "cd3d_45_slabs9")
    return request.param, P, o


def test_reduced_solve_matches_dense_solve(chain):
    name, P, o = chain
    if name == "cd3d_45_slabs9":
        pytest.skip("oracle G^ not formed for this size (full solve checked below)")
    S = make_solver(P, **FP64_DIRECT)
    for seed in (1, 2):
        g = np.random.default_rng(seed).standard_normal(o.m)
        z = host(S.reduced_solve(dev(g)))
        zo, _ = o.reduced_solve(g, mode="direct")
        # FP32 block LU of a G^ whose condition number is modest (M-matrices)
        assert relerr(z, zo) <= 1e-4, (name, seed)
    S.close()


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_full_solve_with_direct_reduced_solve(chain, form):
    name, P, o = chain
    opts = FP64_DIRECT if form == "fp64" else MIXED_DIRECT
    S = make_solver(P, tol_out=1e-12, **opts)
    x, info = S.solve(dev(P.f))
    assert info["status"] == "DDPS_OK", info
    assert info["inner_iterations"] == 0
    x = host(x)
    assert np.max(np.abs(P.f - o.A @ x)) / np.max(np.abs(P.f)) <= 1e-12
    xo = np.linalg.solve(o.A.toarray(), P.f) if P.n <= 5000 else P.x_true
    assert relerr(x, xo) <= 1e-8, name
    S.close()


def test_direct_precond_is_the_exact_preconditioner_to_fp32():
    """Fig. 3 with the direct reduced solve equals the oracle's P^-1 y (direct
    mode) to FP32 accuracy, so the outer iteration needs at most 1.5 steps."""
    P = W.small_convdiff_3d(12, [3, 5, 4])
    o = DDPSOracle(P.n, P.rowptr, P.colind, P.values, P.block_ptr)
    S = make_solver(P, **FP64_DIRECT)
    y = np.random.default_rng(3).standard_normal(P.n)
    z = host(S.precond_apply(dev(y)))
    zo, _ = o.precond(y, mode="direct")
    assert relerr(z, zo) <= 1e-4
    x, info = S.solve(dev(P.f))
    assert info["outer_iterations"] <= 1.5


def test_direct_on_a_batch_of_chains():
    """Systems of different sizes stacked in one handle: one block LU per
    system, all systems' chain steps in the same launches."""
    probs = [W.small_convdiff_2d(N_, 8, seed=k) for k, N_ in enumerate([40, 33, 57, 24])]
    S = Solver.from_systems([(p.rowptr, p.colind, p.values, p.block_ptr) for p in probs],
                            tol_out=1e-12, **MIXED_DIRECT)
    S.factor(dev(S.values_host))
    x, info = S.solve(dev(np.concatenate([p.f for p in probs])))
    assert info["status"] == "DDPS_OK" and info["inner_iterations"] == 0
    x = host(x)
    for k, p in enumerate(probs):
        o = DDPSOracle(p.n, p.rowptr, p.colind, p.values, p.block_ptr, spikes=False)
        xo = np.linalg.solve(o.A.toarray(), p.f)
        assert relerr(x[S.sys_row_ptr[k]:S.sys_row_ptr[k + 1]], xo) <= 1e-8, k
    S.close()


def test_direct_rejects_partitions_that_are_not_chains():
    P = W.small_random_dd(301, 7, seed=9)  # random couplings between any blocks
    with pytest.raises(N.DDPSError, match="INVALID_ARG.*chain"):
        Solver(P.rowptr, P.colind, P.block_ptr, **FP64_DIRECT)
    Q = W.small_convdiff_2d(24, 3)
    with pytest.raises(N.DDPSError, match="INVALID_ARG.*EXPLICIT"):
        Solver(Q.rowptr, Q.colind, Q.block_ptr, ghat_mode=N.DDPS_GHAT_IMPLICIT,
               **{k: v for k, v in FP64_DIRECT.items()})


@pytest.mark.parametrize("name,make", [
    ("one_step", lambda: W.small_convdiff_2d(21, 3)),          # 21 columns: part of a 32-column stage
    ("two_steps", lambda: W.small_convdiff_2d(97, 4)),         # Gauss-Jordan steps of 64 and 33
    ("odd_planes", lambda: W.small_convdiff_3d(13, [4, 5, 4])),  # 169 columns, rows not 16-byte aligned
    ("tiles", lambda: W.small_convdiff_3d(20, [5, 5, 5, 5])),  # 400 columns: ragged 128 x 128 tiles
])
def test_block_lu_on_the_stored_matrix(name, make):
    """The direct reduced solve satisfies the stored G^ in FP64 to FP32 accuracy: the block
    LU's products of up to 800 terms round to about 1e-6, 1e-5 bounds it."""
    P = make()
    S = make_solver(P, **MIXED_DIRECT)
    g = np.random.default_rng(2).uniform(-1, 1, S.m)
    z = host(S.reduced_solve(dev(g)))
    r = g - z
    for b in range(P.p):
        q0, q1, cols = S.ghat_layout(b)
        r[q0:q1] -= S.ghat_block(b) @ z[cols]
    assert np.linalg.norm(r) <= 1e-5 * np.linalg.norm(g), name
    S.close()


def _fp32_block_elimination(G, q, rhs):
    """The block elimination of a chain's reduced system, all in FP32: S_0 = I,
    S_b = I - L_b S_{b-1}^-1 U_{b-1}, inverses by Gauss-Jordan steps without exchanges."""
    f = np.float32
    p = len(q) - 1
    blk = lambda i, j: G[q[i]:q[i + 1], q[j]:q[j + 1]].astype(f)

    def inverse(S):
        S = S.copy()
        for j in range(len(S)):
            piv, row, col = f(1) / S[j, j], S[j].copy(), S[:, j].copy()
            row *= piv
            col[j] = 0
            S[:, j] = 0
            S[j] = 0
            S -= np.outer(col, row)
            S[j] = row
            S[:, j] = -col * piv
            S[j, j] = piv
        return S
    inv = [np.eye(q[1] - q[0], dtype=f)]
    for b in range(1, p):
        inv.append(inverse(np.eye(q[b + 1] - q[b], dtype=f) - blk(b, b - 1) @ (inv[-1] @ blk(b - 1, b))))
    y = [rhs[q[0]:q[1]].astype(f)]
    for b in range(1, p):
        y.append(rhs[q[b]:q[b + 1]].astype(f) - blk(b, b - 1) @ (inv[b - 1] @ y[-1]))
    z = [inv[-1] @ y[-1]]
    for b in range(p - 2, -1, -1):
        z.insert(0, inv[b] @ (y[b] - blk(b, b + 1) @ z[0]))
    return np.concatenate(z)


@pytest.mark.parametrize("side,p", [(24, 3), (33, 5), (47, 9), (64, 4), (97, 6), (128, 7)])
def test_direct_reduced_solve_is_as_exact_as_fp32(side, p):
    """Rounding errors of the products must not add up in one direction: the error of reduced
    solves against FP64, over 24 right-hand sides, is that of an elimination in FP32 (half as
    much again for the scatter between two orders of summation)."""
    P = W.small_convdiff_2d(side, p, seed=side)
    S = make_solver(P, factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3, ghat_prec=N.DDPS_FP32,
                    inner_prec=N.DDPS_FP32, reduced_solver=N.DDPS_REDUCED_DIRECT)
    G, q = np.eye(S.m), [0]
    for b in range(p):
        q0, q1, cols = S.ghat_layout(b)
        G[q0:q1, cols] += S.ghat_block(b)
        q.append(q1)
    rng = np.random.default_rng(side)
    here, ref = [], []
    for _ in range(24):
        g = rng.uniform(-1, 1, S.m)
        z = np.linalg.solve(G, g)
        here.append(relerr(host(S.reduced_solve(dev(g))), z))
        ref.append(relerr(_fp32_block_elimination(G, q, g).astype(np.float64), z))
    rms = lambda v: np.sqrt(np.mean(np.square(v)))
    assert rms(here) <= 1.5 * rms(ref), (rms(here), rms(ref))
    S.close()
