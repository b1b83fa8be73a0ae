"""A training step whose GEMM reported a timeout is not made: the parameters and Adam's step count stay as they were,
and the next call says so, also when the step itself was queued without asking for its loss.  The flag is set by the
host here (no kernel fails): the network's source is compiled into a library of its own with a setter beside it."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
SRC = """
#include "mlp.cu"
namespace sscs { void record_error(const char*) {} }
extern "C" void set_err(scs_mlp* n)
{
    const int one = 1;
    cudaMemcpy(n->err, &one, sizeof one, cudaMemcpyHostToDevice);
}
extern "C" int step_count(scs_mlp* n) { return n->step; }
"""

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("mlp")
    (d / "mlp_flag.cu").write_text(SRC)
    so = str(d / "mlp_flag.so")
    subprocess.run([NVCC, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-diag-suppress", "177", "-shared", "-Xcompiler", "-fPIC", "-cudart",
                    "shared", "-I",
                    os.path.join(ROOT, "paper_1903_06477_gb300", "csrc"), "-o", so, str(d / "mlp_flag.cu")], check=True)
    return C.CDLL(so)


def test_steps_behind_an_error_are_reported_and_do_not_count(lib):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(4)
    X = torch.as_tensor(rng.standard_normal((32, 40)).astype(np.float32), device="cuda")
    T = torch.as_tensor(rng.standard_normal((32, 50)).astype(np.float32), device="cuda")
    out = torch.empty(32, 50, device="cuda")
    torch.cuda.synchronize()
    p = [C.c_void_p(t.data_ptr()) for t in (X, T, out)]
    nets = []
    for _ in range(2):
        h = C.c_void_p()
        assert lib.scs_mlp_create(40, 64, 50, 64, C.c_uint64(3), None, C.byref(h)) == 0
        nets.append(h)

    def step(h, loss=None):
        return lib.scs_mlp_train_step(h, p[0], p[1], 32, C.c_float(0.01), loss)

    def params(h):
        lib.scs_mlp_num_params.restype = C.c_int64
        a = np.empty(lib.scs_mlp_num_params(h), np.float32)
        assert lib.scs_mlp_get_params(h, C.c_void_p(a.ctypes.data)) == 0
        return a

    a, b = nets
    loss = C.c_float(-1.0)
    assert step(a) == 0 and step(b) == 0
    one = params(a)
    for again in (lambda: step(a), lambda: lib.scs_mlp_forward(a, p[0], 32, p[2]),
                  lambda: step(a, C.byref(loss)), lambda: lib.scs_mlp_gradients(a, p[0], p[1], 32, None, C.byref(loss))):
        torch.cuda.synchronize()
        lib.set_err(a)
        assert step(a) == 0  # queued; skipped on the device
        torch.cuda.synchronize()
        assert again() != 0  # reported by the next call, whichever it is
        assert lib.step_count(a) == 1
        assert np.array_equal(params(a), one)
    lib.set_err(a)
    assert step(a, C.byref(loss)) != 0  # a step that waits reports its own
    assert lib.step_count(a) == 1 and np.array_equal(params(a), one)
    assert step(a, C.byref(loss)) == 0 and step(b, C.byref(loss)) == 0
    assert lib.step_count(a) == 2 and np.array_equal(params(a), params(b))
    for h in nets:
        lib.scs_mlp_destroy(h)
