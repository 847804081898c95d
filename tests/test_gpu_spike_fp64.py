"""FP64 spike products: G^ of a block whose rows are all interface rows, by its residual
M X = R, over sizes at the edges of the 32-row and 128-column tiles and of longer sums, with
unknowns and equations in very different units (powers of two, so that they change no
rounding), with couplings that are numerically nothing, and the relative error of its small
entries."""

import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import dev
from paper_1008_1700_gb300 import Solver, native as N

pytestmark = pytest.mark.gpu

FP64 = dict(factor_prec=N.DDPS_FP64, spike_prec=N.DDPS_FP64, ghat_prec=N.DDPS_FP64,
            inner_prec=N.DDPS_FP64)


def _block(kind, size, rng):
    if kind == "dense":
        M = rng.uniform(-1.0, 1.0, (size, size))
    else:  # 7-point grid of size^3: a tree of fronts, with L21 and U12 products
        def line(k):
            return sp.diags([1.0] * 2, [-1, 1], shape=(k, k))
        e = sp.identity(size)
        P = (sp.kron(sp.kron(line(size), e), e) + sp.kron(sp.kron(e, line(size)), e)
             + sp.kron(sp.kron(e, e), line(size)))
        M = P.toarray() * rng.uniform(-1.0, 1.0, P.shape)
    np.fill_diagonal(M, 0.0)
    np.fill_diagonal(M, 1.5 * np.abs(M).sum(axis=1) + 0.1)
    return M


@pytest.mark.parametrize("kind,size,q,units", [
    ("dense", 1, 1, 0), ("dense", 31, 127, 0), ("dense", 33, 128, 12), ("dense", 129, 129, 0),
    ("dense", 160, 5, 12), ("grid", 9, 130, 0), ("grid", 11, 40, 12), ("grid", 11, 1100, 0),
])
def test_ghat_residual(kind, size, q, units):
    rng = np.random.default_rng([size, q, units])
    M = _block(kind, size, rng)
    nb = len(M)
    R = rng.uniform(-1.0, 1.0, (nb, q)) * (rng.random((nb, q)) < (1.0 if kind == "dense" else 0.02))
    R[rng.integers(0, nb, q), np.arange(q)] = 1.0  # every column couples
    C = 0.01 * rng.uniform(0.5, 1.0, (q, nb)) * (rng.random((q, nb)) < 0.05)
    C[rng.integers(0, q, nb), np.arange(nb)] = 0.01  # every row of the block is in the interface
    A = np.block([[M, R], [C, np.eye(q) * 10.0]])
    # 2^(d1_i + d2_j): the exact solution's entries change by powers of two alone
    d1, d2 = (rng.integers(-units, units + 1, nb + q) for _ in range(2))
    S_ = sp.csr_matrix(np.ldexp(A, d1[:, None] + d2[None, :]))
    S_.sort_indices()
    S = Solver(S_.indptr, S_.indices, np.array([0, nb, nb + q]), **FP64)
    S.factor(dev(S_.data))
    q0, q1, cols = S.ghat_layout(0)
    c = S.interface()
    assert (q0, q1) == (0, nb) and np.array_equal(c[q0:q1], np.arange(nb))
    X = np.zeros((nb, q))
    X[:, c[cols] - nb] = np.ldexp(S.ghat_block(0), d2[:nb, None] - d2[c[cols]][None, :])
    res = np.longdouble(M) @ X - R
    # LU without exchanges of a diagonally dominant matrix: |L||U| <= 3 |M|, n roundings each
    # for the factors and the two triangular products, by columns
    bound = 3 * 3 * nb * 2.0 ** -53 * np.linalg.norm(np.abs(M) @ np.abs(X), axis=0)
    assert np.all(np.linalg.norm(res.astype(float), axis=0) <= bound)
    S.close()


def _ghat(M, R):
    """G^ = M^-1 R of a block whose rows are all interface rows; R: one column per coupling
    unknown, with an entry in every column."""
    nb, q = R.shape
    C = np.zeros((q, nb))
    C[np.arange(nb) % q, np.arange(nb)] = 0.01
    A = sp.csr_matrix(np.block([[M, R], [C, np.eye(q) * 10.0]]))
    A.sort_indices()
    S = Solver(A.indptr, A.indices, np.array([0, nb, nb + q]), **FP64)
    S.factor(dev(A.data))
    q0, q1, cols = S.ghat_layout(0)
    c = S.interface()
    assert (q0, q1) == (0, nb) and np.array_equal(c[q0:q1], np.arange(nb))
    X = np.zeros((nb, q))
    X[:, c[cols] - nb] = S.ghat_block(0)
    S.close()
    return X


@pytest.mark.parametrize("weak", [1e-12, 1e-17, 1e-40, 1e-300])
@pytest.mark.parametrize("kind", ["half", "band"])
def test_weak_couplings_in_part_of_a_block(kind, weak):
    """Couplings that are numerically nothing, in half of the rows or far from the diagonal,
    cost the other rows no digits."""
    rng = np.random.default_rng(7)
    nb, q = 130, 140
    M = rng.uniform(-1.0, 1.0, (nb, nb))
    if kind == "half":
        M[nb // 2:] *= weak
    else:
        far = np.abs(np.subtract.outer(np.arange(nb), np.arange(nb)))
        M[far > 3] *= weak
    np.fill_diagonal(M, 0.0)
    np.fill_diagonal(M, 1.5 * np.abs(M).sum(axis=1) + 1.0)
    R = rng.uniform(-1.0, 1.0, (nb, q))
    X = _ghat(M, R)
    res = np.longdouble(M) @ X - R
    # as in test_ghat_residual
    bound = 3 * 3 * nb * 2.0 ** -53 * np.linalg.norm(np.abs(M) @ np.abs(X), axis=0)
    assert np.all(np.linalg.norm(res.astype(float), axis=0) <= bound)


def test_small_entries_keep_their_digits():
    """A strongly dominant M-matrix on a 7-point grid: every sum of the factorisation and of
    the sweeps has terms of one sign but for the pivots, which lose a few percent, so each
    entry of G^ carries a relative error of the roundings it passed through, at most nb in
    each of the LU, the inverses and the two sweeps -- also where it is 2^-140 of the
    column's largest."""
    n1 = 7
    line = sp.diags([1.0] * 2, [-1, 1], shape=(n1, n1))
    e = sp.identity(n1)
    P = (sp.kron(sp.kron(line, e), e) + sp.kron(sp.kron(e, line), e) + sp.kron(sp.kron(e, e), line))
    rng = np.random.default_rng(3)
    M = -P.toarray() * rng.uniform(0.5, 1.0, P.shape) * 2.0 ** -7 + np.eye(n1 ** 3)
    nb, q = len(M), 40
    R = np.zeros((nb, q))
    R[rng.choice(nb, q, replace=False), np.arange(q)] = 1.0
    X = _ghat(M, R)
    W = np.concatenate([M, R], axis=1).astype(np.longdouble)
    for j in range(nb):  # Gauss-Jordan without exchanges: entries of one sign here too
        W[j] /= W[j, j]
        col = W[:, j].copy()
        col[j] = 0
        W -= np.outer(col, W[j])
    ref = W[:, nb:]
    assert ref.min() > 0 and float(ref.min()) < 2.0 ** -100
    assert np.max(np.abs(X - ref) / ref) <= 1.2 * 4 * (nb + 1) * 2.0 ** -53


def test_overflowed_inverse_is_not_a_number():
    """An equation in units of 1e-310, eliminated last: its pivot passes the test against the
    row's norm, but the pivot's reciprocal overflows.  G^ is not finite there."""
    rng = np.random.default_rng(5)
    nb, q = 8, 3
    M = rng.uniform(-1.0, 1.0, (nb, nb))
    np.fill_diagonal(M, 10.0)
    R = rng.uniform(0.5, 1.0, (nb, q))
    C = np.full((q, nb), 0.01)
    rows = sp.csr_matrix(np.block([[M, R], [C, np.eye(q) * 10.0]]))
    _, perm, _ = N.ddps_symbolic(rows.indptr, rows.indices, np.array([0, nb, nb + q]),
                                 values=rows.data, options=N.default_options(**FP64))
    last = int(perm[nb - 1])
    M[last] *= 1e-310
    R[last] *= 1e-310
    X = _ghat(M, R)
    assert not np.isfinite(X[last]).any()
