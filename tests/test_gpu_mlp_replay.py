"""A training step captured in a CUDA graph updates the weights at every replay, without the host: the transposed
weight copies of the backward pass (legacy kernel) and of scs_mlp_read must follow the weights all the same."""
import numpy as np
import pytest

from paper_1903_06477_gb300 import binding as B
from test_gpu_mlp import check_gemm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gemm", [B.GEMM_MMA, B.GEMM_TCGEN05])
def test_transposed_weights_follow_replays(gemm):
    torch = pytest.importorskip("torch")
    dims, batch = (40, 64, 50), 32
    rng = np.random.default_rng(6)
    X = torch.as_tensor(rng.standard_normal((batch, dims[0])).astype(np.float32), device="cuda")
    T = torch.as_tensor(rng.standard_normal((batch, dims[2])).astype(np.float32), device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    net = B.MLP(*dims, max_batch=64, seed=3, stream=stream, gemm=gemm)
    net.gradients(X, T)  # (a step outside the graph has made the copies)

    def step():
        assert B.lib().scs_mlp_train_step(net.h, B._ptr(X), B._ptr(T), batch, 0.05, None) == 0

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        step()
    for _ in range(3):
        before = {k: net.read(k) for k in ("w2", "w3", "w2t", "w3t")}
        assert np.array_equal(before["w2t"], before["w2"].T) and np.array_equal(before["w3t"], before["w3"].T)
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        assert not np.array_equal(net.read("w3"), before["w3"])
        check_gemm("dh2", net.read("dh2"), net.read("dy16"), before["w3"].T, mask=net.read("h2"))
        check_gemm("dh1", net.read("dh1"), net.read("dh2_16"), before["w2"].T, mask=net.read("h1"))
    net.close()
