"""The column-blocked layout where the lanes of a row differ from segment to segment: rows from one entry to thousands
beside one another, a warp a row, one and many column blocks, rows and segments without entries.

The host check replays the product over the layout (scs_cb_layout_check); on the GPU the product itself is compared
with the CSR product.  Bound as for the other layouts: |y - A x| <= gamma_k |A||x|, k the longest row plus the lanes'
and segments' extra additions (below 64), u the unit roundoff of the precision the product ran in."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1903_06477_gb300 import binding as B


def _rows(lens, cols, seed=0):
    """A CSR matrix whose row i has lens[i] entries at random distinct columns."""
    rng = np.random.default_rng(seed)
    idx = [np.sort(rng.choice(cols, k, replace=False)) for k in lens]
    ptr = np.concatenate([[0], np.cumsum(lens)])
    ind = np.concatenate(idx) if ptr[-1] else np.zeros(0, int)
    return sp.csr_matrix((rng.standard_normal(ptr[-1]), ind, ptr), shape=(len(lens), cols))


def _family(name):
    rng = np.random.default_rng(1)
    if name == "long":  # a warp a row: 7, 8, 9 and more steps of 32, with remainders
        return _rows([223, 225, 256, 257, 289, 0, 1025, 5000] * 30 + [3] * 500, 6000)
    if name == "mixed":  # long rows beside short ones, so that both ends of the choice of lanes occur
        return _rows(list(rng.choice([1, 2, 3, 700, 2000], 900)), 2500)
    if name == "wide":  # many column blocks, most segments with few entries, some with none
        return _rows(list(rng.integers(0, 40, 9000)), 70001)
    return _rows([1] * 300 + [0] * 20 + [2] * 7, 11)  # "narrow"


NAMES = ["long", "mixed", "wide", "narrow"]


@pytest.mark.parametrize("elem_bytes", [4, 8])
@pytest.mark.parametrize("warps,vectors,smem", [(15, 1, 209536), (15, 2, 209536), (3, 1, 120000), (1, 2, 209536)])
@pytest.mark.parametrize("name", NAMES)
def test_replay(name, warps, vectors, smem, elem_bytes):
    A = _family(name)
    x = np.random.default_rng(2).standard_normal(A.shape[1])
    y, st = B.cb_layout_check(A, x, compute_warps=warps, elem_bytes=elem_bytes, vectors=vectors, smem_bytes=smem)
    assert st["column_blocks"] > 0 and st["violations"] == 0 and st["smem_bytes"] <= smem
    k = int(np.diff(A.indptr).max()) + 64
    assert np.all(np.abs(y - A @ x) <= k * 2.0**-53 / (1 - k * 2.0**-53) * (abs(A) @ np.abs(x)))


@pytest.mark.gpu
@pytest.mark.parametrize("threads", [0, 64, 160])
@pytest.mark.parametrize("name", NAMES)
def test_product(name, threads):
    A = _family(name)
    m, n = A.shape
    prob = dict(A=A, b=np.ones(m), c=np.ones(n), f=0, l=m, q=[], s=[])
    w = B.Work(prob, team=B.TEAM_GRID, precision=B.MIXED, spmv_path=3, threads=threads, cg_max=1)
    rng = np.random.default_rng(3)
    absA = abs(A)
    for M, absM, op in ((A, absA, 0), (A.T.tocsr(), absA.T.tocsr(), 1), (A.T.tocsr(), absA.T.tocsr(), 2)):
        k = int(np.diff(M.indptr).max()) + 64
        for precision, u in ((B.FP64, 2.0**-53), (B.MIXED, 2.0**-24)):
            xs = [rng.standard_normal(M.shape[1]) for _ in range(2 if op == 2 else 1)]
            ys = w.spmv(xs[0], op, precision, v2=xs[-1])
            for x, y in zip(xs, ys if op == 2 else [ys]):
                # FP32: the inputs and the matrix are rounded too (two more roundings a term)
                g = (k + 3) * u / (1 - (k + 3) * u)
                assert np.all(np.abs(y - M @ x) <= g * (absM @ np.abs(x)))
    w.close()
