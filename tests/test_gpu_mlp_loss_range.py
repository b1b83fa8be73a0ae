"""The network's loss over the range of errors: squares beyond FP32 (an error of 1.9e19 and more), infinities and NaN
give what the FP64 sum of the squares gives, ordinary errors beside them included.  The squares and their sum carry at
least 48 bits, so what is left is the rounding of the loss to FP32 (and of the errors themselves: y and the target are
subtracted in FP32 on both sides here)."""
import numpy as np
import pytest

from paper_1903_06477_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gemm", [B.GEMM_TCGEN05, B.GEMM_MMA])
@pytest.mark.parametrize("d_out", [36, 37])  # rows at multiples of 16 bytes, and not
@pytest.mark.parametrize("value", [1.0, 1e10, 1.8e19, 2.5e19, -1e20, np.inf, -np.inf, np.nan])
def test_loss_of_large_errors(value, d_out, gemm):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(d_out)
    net = B.MLP(24, 32, d_out, max_batch=32, seed=2, gemm=gemm)  # never fitted: mean 0, deviation 1
    X = rng.standard_normal((20, 24)).astype(np.float32)
    T = rng.standard_normal((20, d_out)).astype(np.float32)
    T[3, 7] = value
    T[19, d_out - 1] = value
    loss = net.gradients(torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda"))
    diff = (net.read("y") - T).astype(np.float64)
    ref = 0.5 * np.mean(diff ** 2)
    if np.isnan(ref):
        assert np.isnan(loss)
    elif np.isinf(ref):
        assert loss == np.inf
    else:
        assert abs(loss - ref) <= 2.0 ** -23 * ref, (loss, ref)
    net.close()
