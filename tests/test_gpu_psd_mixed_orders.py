"""PSD blocks above and below order 64 in one problem: the larger ones are decomposed in global memory, the smaller
ones beside them in shared memory.  Pi_C against the FP64 oracle with the bounds of the parity tests: 1e-10 in FP64,
1e-4 ||X||_F as the FP32 phase runs it, 6 units of FP32 rounding with every block redone in FP64."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1903_06477_gb300 import binding as B
from paper_1903_06477_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("team", [B.TEAM_BLOCK, B.TEAM_GRID])
@pytest.mark.parametrize("psd", [[65, 64], [100, 41, 64], [120, 60], [80, 33, 20], [65, 13], [20, 151, 64, 7, 48, 66]])
def test_projection_across_order_64(psd, team):
    prob = W.planted(seed=45, n=30, l=7, psd=psd, nnz=3000)
    orc = O.Oracle(prob)
    off = np.cumsum([30 + 7] + [d * (d + 1) // 2 for d in psd])
    rng = np.random.default_rng(11)
    v = rng.standard_normal(off[-1] + 1) * 2
    default = B.Work(prob, team=team, precision=B.MIXED)
    forced = B.Work(prob, team=team, precision=B.MIXED, psd_recheck_tol=0.0)
    plain = B.Work(prob, team=team)  # no FP32 kernels: its launches have the FP64 need alone
    for _ in range(2):  # the second pass starts from the first one's eigenvectors
        ref = orc.proj_C(v)
        for w in (default, plain):
            np.testing.assert_allclose(w.project_cone(v), ref, rtol=0, atol=1e-10)
        out, _ = default.project_cone_prec(v, B.MIXED)
        redone, stats = forced.project_cone_prec(v, B.MIXED)
        assert stats[1] == len(psd)
        for o, e in zip(off[:-1], off[1:]):
            size = np.linalg.norm(v[o:e])
            assert np.linalg.norm(out[o:e] - ref[o:e]) <= 1e-4 * size
            assert np.linalg.norm(redone[o:e] - ref[o:e]) <= 6 * 2.0 ** -24 * size
        v = v + 0.03 * rng.standard_normal(v.size)
    for w in (default, forced, plain):
        w.close()
