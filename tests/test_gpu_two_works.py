"""Works and batches of different shared-memory needs alive at the same time: the kernels' limit belongs
to the function, so a later, smaller setup must not refuse an earlier, larger work its launches."""
import numpy as np
import pytest

from paper_1903_06477_gb300 import binding as B
from paper_1903_06477_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [B.FP64, B.MIXED])
@pytest.mark.parametrize("team", [B.TEAM_BLOCK, B.TEAM_GRID])
def test_larger_work_still_runs_after_a_smaller_setup(team, precision):
    big = W.planted(seed=1, n=30, l=5, psd=[64], nnz=500)
    works = [B.Work(W.planted(seed=s, n=30, l=5, psd=[d], nnz=200), team=team, precision=precision)
             for s, d in ((2, 20), (3, 41))]
    first = B.Work(big, team=team, precision=precision)
    rng = np.random.default_rng(0)
    v = rng.standard_normal(first.N)
    before = first.project_cone(v)
    works += [B.Work(W.planted(seed=s, n=30, l=5, psd=[d], nnz=200), team=team, precision=precision)
              for s, d in ((4, 33), (5, 2))]
    works.append(B.Work(W.planted(seed=6, n=20, l=30, nnz=100), team=team, precision=precision))
    # the same projection, from the eigenvectors of the first one
    assert np.allclose(first.project_cone(v), before, rtol=0, atol=1e-12 * (1 + np.abs(before).max()))
    for w in works:
        assert np.isfinite(w.project_cone(rng.standard_normal(w.N))).all()
    for w in works + [first]:
        w.close()
