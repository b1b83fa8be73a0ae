"""The direct linear solves (one thread block, linsys_direct): (I + Q)^{-1} r at
the edges of the inversion's 32 x 32 tiles and of the solve's split of the rows
over idle warps, against a dense FP64 solve of the same system."""
import numpy as np
import pytest

from paper_1903_06477_gb300 import binding as B
from paper_1903_06477_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [32, 128, 256, 1024])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 97, 128, 129, 257, 400])
def test_direct_linsys_matches_dense_solve(n, threads):
    prob = W.planted(seed=n, n=n, l=n + 7, soc=(5, 9), nnz=min(n * (n + 21), 12 * n + 20))
    work = B.Work(prob, team=B.TEAM_BLOCK, threads=threads, linsys_direct=1)
    A, h = prob["A"].toarray(), np.concatenate([prob["c"], prob["b"]])
    m = A.shape[0]
    K = np.block([[np.eye(n), A.T, prob["c"][:, None]], [-A, np.eye(m), prob["b"][:, None]],
                  [-h[None, :], np.ones((1, 1))]])
    rng = np.random.default_rng(n + threads)
    # the inverse's error is a few n u cond(I + A^T A) of the x part, carried to y by A and to all by tau
    cond = 1.0 + np.linalg.norm(A, 2) ** 2
    for _ in range(3):  # the second and third start from the last solution
        r = rng.standard_normal(n + m + 1)
        ref = np.linalg.solve(K, r)
        out = work.linsys(r)
        assert np.linalg.norm(out - ref) <= 100 * (n + m) * 2.2e-16 * cond * (1 + np.linalg.norm(h)) * np.linalg.norm(ref)
    work.close()
