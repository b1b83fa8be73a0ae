"""Shared memory of the PSD projections (host code, no GPU): what psd_plan hands a group of threads must hold every
block of the problem as psd_layout places it.  The need is not monotone in the order -- above order 64 a block's
matrices are in global memory -- so the largest order alone does not size it.  Group bytes and layout come from the
same header, compiled for the host; the end of a block's layout is worked out here from its pointers."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
SRC = """
#include "solver.cuh"
using namespace sscs;
template <typename T>
static void check(int n, const int* orders, int ctas, int threads, long* out)
{
    int order, small;
    psd_orders(std::vector<int>(orders, orders + n), order, small);
    const PsdPlan p = psd_plan<T>(order, small, n, ctas, threads, 200 * 1024);
    unsigned char* base = (unsigned char*)(1ul << 20);
    unsigned char* big = (unsigned char*)(1ul << 40);
    long end = 0;
    for (int i = 0; i < n; ++i) {
        const int d = orders[i], dp = d + (d & 1);
        const PsdSmem<T> s = psd_layout<T>(base, d > PSD_MAX ? big : nullptr, dp);
        const size_t full = sizeof(T) * dp * (dp + 1), cells = sizeof(T) * 4 * Jacobi<T>::cells(dp);
        const unsigned char* ends[] = {(unsigned char*)(s.red + 33),
                                       (unsigned char*)(s.scratch + Jacobi<T>::scratch_words(dp)),
                                       (unsigned char*)s.lam + sizeof(double) * dp,  // FP64 eigenvalues of a redo
                                       (unsigned char*)s.X0 + full, (unsigned char*)s.V + full,
                                       (unsigned char*)s.V + sizeof(T) * dp * psd_ldv<T>(dp),
                                       (unsigned char*)s.cell[0] + cells, (unsigned char*)s.cell[1] + cells,
                                       sizeof(T) == 4 ? (unsigned char*)s.V64 + 8 * dp * (dp + 1) : base};
        for (const unsigned char* e : ends)
            if (e < big && e - base > end) end = e - base;
    }
    out[0] = p.bytes;
    out[1] = p.groups;
    out[2] = p.threads;
    out[3] = end;
}
extern "C" void plan(int n, const int* orders, int ctas, int threads, int esize, long* out)
{
    esize == 8 ? check<double>(n, orders, ctas, threads, out) : check<float>(n, orders, ctas, threads, out);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("psd_plan")
    (d / "plan.cu").write_text(SRC)
    so = str(d / "plan.so")
    subprocess.run([NVCC, "-O0", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared", "-I",
                    os.path.join(ROOT, "paper_1903_06477_gb300", "csrc"), "-o", so, str(d / "plan.cu")], check=True)
    fn = C.CDLL(so).plan

    def run(orders, ctas, threads, esize):
        a, out = np.array(orders, np.int32), np.zeros(4, np.int64)
        fn(len(a), C.c_void_p(a.ctypes.data), ctas, threads, esize, C.c_void_p(out.ctypes.data))
        return [int(x) for x in out]

    return run


MIXES = [[120, 60], [65, 13], [65, 64], [100, 41], [80, 33, 20], [151, 64, 7], [65, 100, 151, 7], [1024, 64],
         [120, 19], [120, 18], [64], [65], [1], [20] * 500, [63, 64] * 200, [1, 2, 64, 3] * 100, [200] * 3 + [48] * 400]


@pytest.mark.parametrize("esize", [8, 4])
@pytest.mark.parametrize("ctas,threads", [(152, 512), (152, 256), (1, 256), (1, 1024), (608, 128), (1, 96)])
def test_plan_holds_every_block(plan, ctas, threads, esize):
    for orders in MIXES + [[big, d] for big in (65, 66, 119, 300) for d in range(1, 65)]:
        size, groups, t, end = plan(orders, ctas, threads, esize)
        assert end <= size, (orders[:4], size, end)
        assert size % 16 == 0 and groups * t <= threads
        assert groups == 1 or groups * size <= 200 * 1024
