"""The direct linear solves (linsys_direct) on ill-conditioned matrices, against triangular solves: the residual that
(I + Q)^{-1} r leaves in the rows x + A^T y + c tau, for r and c in the range of A^T as a solver's are, is compared with
that of the same elimination done with numpy's Cholesky factor of the same matrix.  With the inverse of the factor it
is a few times that one (a simulation in numpy, 20 to 300 columns: 1.4 to 4.5 times); with the inverse of the whole
matrix it was 800 to 110 000 times.  The line is drawn at 32.  Each system is solved by a work of its own: a solve starts from
the last solution, and the rounding of that start is not what is compared."""
import numpy as np
import pytest
import scipy.linalg as sl
import scipy.sparse as sp

from paper_1903_06477_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _residual(A, c, e, x, tau):
    A, x = A.astype(np.longdouble), x.astype(np.longdouble)
    return float(np.linalg.norm(-(A.T @ e.astype(np.longdouble)) - c * np.longdouble(tau) - x - A.T @ (A @ x)))


@pytest.mark.parametrize("n,threads", [(20, 256), (33, 256), (50, 32), (120, 1024), (300, 256)])
@pytest.mark.parametrize("log_sigma", [4, 6])
def test_residual_like_triangular_solves(n, threads, log_sigma):
    rng = np.random.default_rng(n + log_sigma)
    m = 2 * n
    U, _ = np.linalg.qr(rng.standard_normal((m, n)))
    V, _ = np.linalg.qr(rng.standard_normal((n, n)))
    A = (U * np.logspace(0, log_sigma, n)) @ V.T  # singular values 1 to 10^log_sigma
    c = -A.T @ rng.standard_normal(m)
    prob = dict(A=sp.csr_matrix(A), b=np.zeros(m), c=c, f=0, l=m, q=[], s=[])
    factor = sl.cho_factor(np.eye(n) + A.T @ A, lower=True)
    g = sl.cho_solve(factor, c)
    here, ref = [], []
    for _ in range(4):
        e = rng.standard_normal(m)
        work = B.Work(prob, team=B.TEAM_BLOCK, threads=threads, linsys_direct=1)
        out = work.linsys(np.concatenate([np.zeros(n), e, [0.0]]))
        work.close()
        here.append(_residual(A, c, e, out[:n], out[-1]))
        x = sl.cho_solve(factor, -(A.T @ e))
        tau = (c @ x) / (1 + c @ g)
        ref.append(_residual(A, c, e, x - tau * g, tau))
    assert np.mean(here) <= 32 * np.mean(ref), (here, ref)
