"""PSD projections of many random blocks against numpy's eigh: each block within what the sweeps' stop leaves, and, from
a cold start in FP64, no further away on average than a cyclic Jacobi iteration with FP64 angles and the same stop.

The sweeps stop at an off-diagonal part of 1e-13 |X| (FP64).  X = V (L + E) V^T with |E| below that, and the projection
is 1-Lipschitz, so a block is within 1e-13 |X| and some roundings of d terms.  Most blocks stop far below: how far is
what the last sweep leaves, which exact angles make quadratically small.  The average is compared with 4 units of
rounding and a tenth to spare for another order of the sums."""
import numpy as np
import pytest

from paper_1903_06477_gb300 import binding as B
from paper_1903_06477_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _mats(v, d):
    """Blocks from their svec rows (count x d (d + 1) / 2)."""
    j, i = np.triu_indices(d)
    X = np.zeros((len(v), d, d))
    X[:, i, j] = v / np.where(i == j, 1.0, np.sqrt(2.0))
    X[:, j, i] = X[:, i, j]
    return X


def _project(X):
    w, V = np.linalg.eigh(X)
    return np.einsum("nik,nk,njk->nij", V, np.maximum(w, 0), V)


def _jacobi(X):
    """Cyclic Jacobi by round-robin pairs, angles in FP64, until the off-diagonal part is 1e-13 of the whole."""
    n, d, _ = X.shape
    dp = d + d % 2
    A = np.zeros((n, dp, dp))
    A[:, :d, :d] = X
    V = np.broadcast_to(np.eye(dp), A.shape).copy()
    mask = ~np.eye(dp, dtype=bool)
    total = (A ** 2).sum((1, 2))
    for _ in range(20):
        live = np.nonzero((A[:, mask] ** 2).sum(1) > 1e-26 * total)[0]
        if not live.size:
            break
        a, v = A[live], V[live]
        for rnd in range(dp - 1):
            k = np.arange(1, dp // 2)
            p, q = np.concatenate([[rnd], (rnd + k) % (dp - 1)]), np.concatenate([[dp - 1], (rnd - k) % (dp - 1)])
            apq, diff = a[:, p, q], a[:, q, q] - a[:, p, p]
            with np.errstate(all="ignore"):
                th = diff / (2 * apq)
                t = np.where(th >= 0, 1.0, -1.0) / (np.abs(th) + np.sqrt(th * th + 1))
            t = np.where(apq == 0, 0.0, t)
            c = 1 / np.sqrt(t * t + 1)
            s = t * c
            for m in (a, v):
                x, y = m[:, :, p].copy(), m[:, :, q].copy()
                m[:, :, p], m[:, :, q] = c[:, None] * x - s[:, None] * y, s[:, None] * x + c[:, None] * y
            x, y = a[:, p, :].copy(), a[:, q, :].copy()
            a[:, p, :], a[:, q, :] = c[:, :, None] * x - s[:, :, None] * y, s[:, :, None] * x + c[:, :, None] * y
        A[live], V[live] = a, v
    w = np.maximum(A[:, np.arange(dp), np.arange(dp)], 0)
    return np.einsum("nik,nk,njk->nij", V, w, V)[:, :d, :d]


@pytest.mark.parametrize("d,count", [(1, 400), (2, 400), (3, 400), (5, 400), (8, 400), (10, 400), (17, 300), (20, 300),
                                     (33, 160), (64, 160), (65, 8)])
def test_blocks_against_eigh(d, count):
    one = d * (d + 1) // 2
    w = B.Work(W.planted(seed=d, n=8, l=0, psd=[d] * count, nnz=one * count), precision=B.MIXED, team=B.TEAM_GRID)
    rng = np.random.default_rng(100 * d)
    v = rng.standard_normal(w.N)
    errors = {}
    for precision in (B.FP64, B.MIXED):
        x = v.copy()
        for warm in (False, True):  # the second pass starts from the first one's eigenvectors
            X = _mats((x if precision == B.FP64 else x.astype(np.float32).astype(float))[8:-1].reshape(count, one), d)
            got = _mats(w.project_cone_prec(x, precision)[0][8:-1].reshape(count, one), d)
            size = np.linalg.norm(X, axis=(1, 2))
            errors[precision, warm] = np.linalg.norm(got - _project(X), axis=(1, 2)) / size
            bound = 1e-13 + 64 * d * U if precision == B.FP64 else 1e-4  # (FP32: the bound of the redo)
            assert errors[precision, warm].max() <= bound, (precision, warm, errors[precision, warm].max())
            if precision == B.FP64 and not warm and d <= 64:
                ref = (np.linalg.norm(_jacobi(X) - _project(X), axis=(1, 2)) / size).mean()
                assert errors[precision, warm].mean() <= 1.1 * ref + 4 * U, (errors[precision, warm].mean(), ref)
            x = x + 0.03 * rng.standard_normal(w.N)
    w.close()
