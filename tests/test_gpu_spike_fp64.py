"""FP64 spike products (fixed-point digits on the tensor cores): G^ of a block whose rows
are all interface rows, by its residual M X = R, over sizes at the edges of the 32-row and
128-column tiles, of the 32-column stages and of the 128-value groups of K, with unknowns
and equations in very different units (powers of two, so that they change no rounding)."""

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
