"""One step of the network on one and two rows (and a few more), stage by stage on each stage's own inputs with the
bounds of test_gpu_mlp: products whose inner or outer size is the number of rows, the ReLU masks, the bias sums and the
Adam update.  The normalisation is fitted to sixteen other rows."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_1903_06477_gb300 import binding as B
from test_gpu_mlp import U, _split, bf16, check_colsum, check_gemm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gemm", [B.GEMM_TCGEN05, B.GEMM_MMA])
@pytest.mark.parametrize("dims", [(33, 40, 17), (129, 136, 999), (8, 8, 8)])
@pytest.mark.parametrize("batch", [1, 2, 7])
def test_stages_of_a_step(dims, batch, gemm):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(sum(dims) + batch)
    fit = [torch.as_tensor(rng.standard_normal((16, d)).astype(np.float32), device="cuda") for d in (dims[0], dims[2])]
    X, T = [rng.standard_normal((batch, d)).astype(np.float32) for d in (dims[0], dims[2])]
    net = B.MLP(*dims, max_batch=64, seed=3, gemm=gemm)
    net.fit_normalization(*fit)
    theta = net.read("params").ravel()
    W1, b1, W2, b2, W3, b3 = _split(theta, dims)
    lr = 2.0 ** -10
    loss = net.train_step(torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda"), lr)
    r = {k: net.read(k).astype(np.float64) for k in B.MLP_BUFFERS}
    w1, w2, w3 = [bf16(W.astype(np.float32)).astype(np.float64) for W in (W1, W2, W3)]
    check_gemm("h1", r["h1"], r["xn"], w1, bias=b1, relu=True, bf16_out=True)
    check_gemm("h2", r["h2"], r["h1"], w2, bias=b2, relu=True, bf16_out=True)
    check_gemm("y", r["y"], r["h2"], w3, bias=b3)
    tn = (T.astype(np.float64) - r["out_mean"]) / r["out_std"]
    diff, scale = r["y"] - tn, 1.0 / (batch * dims[2])
    assert abs(loss - 0.5 * np.mean(diff ** 2)) <= 1e-5 * loss
    bound = 6 * U * (np.abs(r["y"]) + np.abs(tn) + np.abs(r["out_mean"] / r["out_std"])) * scale + 1e-38
    assert (np.abs(r["dy"] - diff * scale) <= bound).all()
    assert np.array_equal(r["dy16"], bf16(r["dy"].astype(np.float32)).astype(np.float64))
    check_gemm("dh2", r["dh2"], r["dy16"], w3.T, mask=r["h2"])
    check_gemm("dh1", r["dh1"], r["dh2_16"], w2.T, mask=r["h1"])
    gW1, gb1, gW2, gb2, gW3, gb3 = _split(r["grad"].ravel(), dims)
    check_gemm("gW3", gW3, r["dy16"].T, r["h2"].T)
    check_gemm("gW2", gW2, r["dh2_16"].T, r["h1"].T)
    check_gemm("gW1", gW1, r["dh1_16"].T, r["xn"].T)
    check_colsum("gb3", gb3, r["dy"])
    check_colsum("gb2", gb2, r["dh2"])
    check_colsum("gb1", gb1, r["dh1"])
    # Adam's first step from zero moments: the moments to a few FP32 roundings, and lr g / (|g| + eps) from them
    g, zero = r["grad"].ravel(), np.zeros(theta.size)
    th, m, v = M.adam_step(theta.astype(np.float64), g, zero, zero, 1, lr)
    assert (np.abs(r["adam_m"].ravel() - m) <= 4 * U * np.abs(g) + 1e-45).all()
    assert (np.abs(r["adam_v"].ravel() - v) <= 6 * U * g * g + 1e-45).all()
    step = np.abs(theta - th)
    dm, dv = np.abs(r["adam_m"].ravel() - m), np.abs(r["adam_v"].ravel() - v)
    b1c, b2c = 1 - 0.9, 1 - 0.999
    den = np.sqrt(v / b2c) + 1e-8
    bound = (U * np.abs(th) + 10 * U * step + lr * (dm + 2 * U * np.abs(m)) / (b1c * den)
             + step * dv / (2 * np.maximum(v, 1e-300)) + 1e-45)
    assert (np.abs(r["params"].ravel() - th) <= bound).all()
    net.close()
