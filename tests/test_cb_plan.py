"""The automatic plan of the column-blocked layout (host code, no GPU): a plan is either whole or absent.
A width that overflows its stage is shrunk and planned again, and the test for too short segments can
then end the plan: what the first attempt had built must not be left behind (a layout with column blocks
but no stage, which the kernel would read and write out of bounds)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest
import scipy.sparse as sp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "cb_layout.h"
extern "C" void plan(int rows, int cols, const int* rp, const int* ci, const double* vx, int esize, int nv, long dyn,
                     long* out)
{
    CbLayout L;
    plan_cb(rows, cols, {rp, rp + rows + 1}, {ci, ci + rp[rows]}, {vx, vx + rp[rows]}, 152, 15, esize, nv, dyn, false, L);
    out[0] = L.ncb;
    out[1] = L.stage_bytes;
    out[2] = (long)L.dyn();
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SRC)
    so = str(d / "plan.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1903_06477_gb300", "csrc"), "-o", so, str(d / "plan.cpp"), "-lpthread"],
                   check=True)
    fn = C.CDLL(so).plan

    def run(M, esize, nv, dyn=209536):
        M = M.tocsr()
        M.sort_indices()
        a = [np.ascontiguousarray(x, t) for x, t in ((M.indptr, np.int32), (M.indices, np.int32), (M.data, np.float64))]
        out = np.zeros(3, np.int64)
        fn(M.shape[0], M.shape[1], *[C.c_void_p(x.ctypes.data) for x in a], esize, nv, C.c_long(dyn),
           C.c_void_p(out.ctypes.data))
        return out, dyn

    return run


def _lasso(n):
    """The rows of the epigraph LASSO with a dense n/5 x n design: 2n rows of two entries, n/5 of n."""
    eye, dense = sp.identity(n, format="csr"), sp.csr_matrix(np.ones((-(-n // 5), n)))
    return sp.vstack([sp.hstack([eye, -eye]), sp.hstack([-eye, -eye]), sp.hstack([dense, 0 * dense])]).tocsr()


@pytest.mark.parametrize("n", [631, 1585, 2300, 2512])
def test_plan_is_whole_or_absent(plan, n):
    A = _lasso(n)
    A.eliminate_zeros()
    for M, nv in ((A, 1), (A.T, 2)):
        for esize in (8, 4):
            (ncb, stage, total), dyn = plan(M, esize, nv)
            assert (ncb == 0) == (stage == 0), (n, nv, esize, ncb, stage)
            assert total <= dyn
