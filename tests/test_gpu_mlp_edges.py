"""The network's GEMMs at the edges of their tiles and ranges, stage by stage on each stage's own inputs (bounds of
test_gpu_mlp): one row, one over and one under a tile of 128 or 256 rows, odd inner and outer sizes (whose rows are
not multiples of 16 bytes), and an inner size long enough for many ranges."""
import numpy as np
import pytest

from paper_1903_06477_gb300 import binding as B
from test_gpu_mlp import run_stages

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,batch", [((33, 40, 17), 1), ((33, 40, 17), 129), ((129, 136, 999), 257),
                                        ((65, 72, 5003), 300), ((1501, 128, 31), 127), ((8, 8, 8), 2)])
def test_stages_at_tile_edges(dims, batch):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(sum(dims) + batch)
    net = B.MLP(*dims, max_batch=max(batch, 64), seed=3, gemm=B.GEMM_TCGEN05)
    rows = max(batch, 16)  # of the data that the normalisation is fitted to
    X = rng.standard_normal((rows, dims[0])).astype(np.float32)
    T = rng.standard_normal((rows, dims[2])).astype(np.float32)
    if batch == rows:
        net.fit_normalization(torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda"))
        run_stages(net, dims, X, T, B.GEMM_TCGEN05)
    else:  # too few rows to fit: the same rows inside a full batch, whose tiles and ranges may differ, so that a
        # hidden value can round the other way (one BF16 unit, 2^-8 of it, in each of two layers)
        net.fit_normalization(torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda"))
        Xd = torch.as_tensor(X, device="cuda")
        full = torch.empty(rows, dims[2], device="cuda")
        few = torch.empty(batch, dims[2], device="cuda")
        net.forward(Xd, full)
        net.forward(Xd[:batch].contiguous(), few)
        assert float((few - full[:batch]).abs().max()) <= 2.0**-7 * float(full.abs().max())
    net.close()
