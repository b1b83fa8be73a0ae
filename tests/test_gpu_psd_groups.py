"""Several PSD blocks at a time in a CTA: copies of the same blocks, spread over the groups of all CTAs, must come out
bit for bit the same whichever group projects them, cold and from the previous eigenvectors (equal work, no tolerance)."""
import numpy as np
import pytest

from paper_1903_06477_gb300 import binding as B
from paper_1903_06477_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pattern,copies,team", [([20], 500, B.TEAM_GRID), ([33], 320, B.TEAM_GRID),
                                                 ([64], 305, B.TEAM_GRID), ([1, 2, 64, 3, 17, 48], 60, B.TEAM_GRID),
                                                 ([24, 7], 9, B.TEAM_BLOCK), ([25, 2], 5, B.TEAM_BLOCK)])
def test_copies_agree(pattern, copies, team):
    one = sum(d * (d + 1) // 2 for d in pattern)
    w = B.Work(W.planted(seed=1, n=8, l=0, psd=pattern * copies, nnz=one * copies), precision=B.MIXED, team=team)
    rng = np.random.default_rng(2)
    block = rng.standard_normal(one)
    v = rng.standard_normal(w.N)
    for precision in (B.FP64, B.MIXED):
        for _ in range(2):
            v[8:-1] = np.tile(block, copies)
            got = w.project_cone_prec(v, precision)[0][8:-1].reshape(copies, one)
            assert np.isfinite(got).all()
            assert (got == got[0]).all()
            block = block + 0.03 * rng.standard_normal(one)
    w.close()
