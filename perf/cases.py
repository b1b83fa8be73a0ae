"""The work the solver library is measured on: what its users have it do, over the range of sizes they have.

Each case is a dict of plain values; `prepare` makes what a user's program holds before the call (the problem data
on the host, the set-up work, batch or network, the buffers), `run` makes the calls.  Problem sizes are those of the
repository's benchmark and of the synthetic families of arXiv 1903.06477 (Sec. 5), and sizes between them.

Whole solves run a fixed budget of outer iterations (`max_iters`, as a caller with a deadline sets it): the iterates
of a fixed budget are a function of the data, while the point at which a tolerance is met moves with the last bit.
Vectors are passed as device buffers where the caller would keep them there (the single operators, the network) and
as host arrays where it would not (whole solves, batches).  Results of an FP32 phase come back from the C ABI widened
to FP64; they are narrowed to FP32 again, which loses nothing.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_1903_06477_gb300 import binding as B
from paper_1903_06477_gb300 import workloads as W

SQRT2 = math.sqrt(2.0)


class Csr:
    """The part of a CSR matrix that the binding reads."""

    def __init__(self, shape, indptr, indices, data):
        self.shape, self.indptr, self.indices, self.data = shape, indptr, indices, data

    @property
    def nnz(self):
        return int(self.indptr[-1])


# ---------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest problem anyone solves: a LASSO of 302 rows, restarted Broyden; all latency
        dict(name="lasso_small", kind="lasso", rows=60, cols=120, density=0.1, direction="rb", iters=20),
        # one instance of the paper's LASSO family (Sec. 5.3): a dense 200 x 1000 design
        dict(name="lasso_paper", kind="lasso", rows=200, cols=1000, density=1.0, direction="aa", iters=20),
        # one instance of the paper's l1-logistic family (Sec. 5.4): 240 exponential cones, linear systems by the
        # dense factor
        dict(name="logreg", kind="logreg", rows=120, cols=100, direction="aa", direct=1, iters=16),
        # one instance of the paper's sparse-PCA family (Sec. 5.2): one PSD block of order 120
        dict(name="sparse_pca", kind="pca", order=120, direction="aa", iters=4),
        # a batch of independent portfolio SOCPs of uneven size, linear systems by the dense factor
        dict(name="portfolio_batch", kind="portfolio", count=1024, low=20, high=400, precision="fp64", iters=20),
        # a batch of LASSO instances that share their design matrix (training data and warm-start runs)
        dict(name="lasso_batch", kind="lasso_batch", count=160, rows=2000, cols=5000, density=0.01, iters=6),
        # the linear systems of one large sparse program, 1e7 nonzeros, FP32 corrections of an FP64 residual: the
        # inner loop of the mixed-precision solve
        dict(name="linsys_mixed", kind="linsys", scale=1.0, precision="mixed"),
        # the first outer iterations of the same program in plain FP64
        dict(name="sparse_solve", kind="sparse_solve", scale=1.0, direction="aa", iters=10),
        # the cone projections of successive iterates of a large SDP as the FP32 phase runs them
        dict(name="sdp_cone_fp32", kind="cone", blocks=512, order_low=64, order_high=64, precision="mixed"),
        # a smaller SDP with blocks of uneven order, whole iterations in FP64
        dict(name="sdp_solve", kind="sdp_solve", blocks=150, order_low=20, order_high=63, direction="aa", iters=6),
        # one training step of the warm-start network
        dict(name="mlp_train", kind="mlp_train", d_in=2000, hidden=1024, d_out=22004, rows=256),
        # the network's inference, as the warm start of a batch of instances
        dict(name="mlp_forward", kind="mlp_forward", d_in=2000, hidden=1024, d_out=22004, rows=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lasso", "logreg", "pca", "portfolio", "lasso_batch", "linsys", "sparse_solve", "cone",
                       "sdp_solve", "mlp_train", "mlp_forward"])
    direction = rng.choice(["aa", "rb", "aa_qr"])
    if kind == "lasso":
        cols = _log(rng, 100, 700)
        return dict(kind=kind, rows=max(20, cols // rng.choice([2, 3, 5])), cols=cols,
                    density=rng.choice([0.1, 0.3, 1.0]), direction=direction, iters=rng.randint(8, 20))
    if kind == "logreg":
        return dict(kind=kind, rows=_log(rng, 30, 120), cols=_log(rng, 30, 100), direction=direction,
                    direct=rng.randint(0, 1), iters=rng.randint(6, 16))
    if kind == "pca":
        return dict(kind=kind, order=_log(rng, 30, 120), direction="aa", iters=4)
    if kind == "portfolio":
        low = rng.randint(20, 120)
        return dict(kind=kind, count=_log(rng, 64, 1024), low=low, high=rng.randint(low + 20, 400), precision="fp64",
                    iters=rng.randint(8, 20))
    if kind == "lasso_batch":
        cols = _log(rng, 500, 5000)
        return dict(kind=kind, count=_log(rng, 32, 160), rows=int(cols * 0.4), cols=cols, density=0.01,
                    iters=rng.randint(3, 6))
    if kind == "linsys":
        return dict(kind=kind, scale=_log(rng, 40, 1000) / 1000.0, precision=rng.choice(["mixed", "fp64"]))
    if kind == "sparse_solve":
        return dict(kind=kind, scale=_log(rng, 40, 900) / 1000.0, direction=direction, iters=rng.randint(5, 10))
    if kind == "cone":
        lo = rng.randint(5, 60)
        return dict(kind=kind, blocks=_log(rng, 16, 512), order_low=lo, order_high=rng.randint(lo, 64),
                    precision=rng.choice(["mixed", "fp64"]))
    if kind == "sdp_solve":
        lo = rng.randint(5, 50)
        return dict(kind=kind, blocks=_log(rng, 16, 150), order_low=lo, order_high=rng.randint(lo, 63),
                    direction="aa", iters=rng.randint(3, 6))
    hidden = 8 * _log(rng, 16, 128)
    return dict(kind=kind, d_in=_log(rng, 100, 2000), hidden=hidden, d_out=_log(rng, 543, 22004),
                rows=_log(rng, 1 if kind == "mlp_forward" else 16, 256))


# ---------------------------------------------------------------------------------------------------------------
# problems, from a seed
# ---------------------------------------------------------------------------------------------------------------
def _sparse(n, m, nnz, seed):
    """A uniform random pattern, which belongs to the sizes, with N(0,1) values from the seed (drawn on the GPU, where
    it takes milliseconds), in host CSR."""
    g = torch.Generator(device="cuda").manual_seed(5)
    key = torch.unique(torch.randint(0, n * m, (nnz,), generator=g, device="cuda", dtype=torch.int64))
    g.manual_seed(seed)
    rows = torch.div(key, n, rounding_mode="floor")
    val = torch.randn(key.numel(), generator=g, device="cuda", dtype=torch.float64).cpu().numpy()
    indptr = np.concatenate([[0], np.cumsum(torch.bincount(rows, minlength=m).cpu().numpy())]).astype(np.int64)
    col = (key - rows * n).to(torch.int32).cpu().numpy()
    return Csr((m, n), indptr, col, val), rows.cpu().numpy()


def _planted(rng, A, rows, l, soc, psd):
    """b and c that give A x + s = b a planted complementary optimum over [l orthant | SOCs | PSD blocks]."""
    m, n = A.shape
    x, s, y = rng.standard_normal(n), np.zeros(m), np.zeros(m)
    pick = rng.random(l) < 0.5
    s[:l] = np.where(pick, rng.uniform(0.1, 1.0, l), 0.0)
    y[:l] = np.where(pick, 0.0, rng.uniform(0.1, 1.0, l))
    o = l
    if soc:
        k, q = len(soc), soc[0]
        u = rng.standard_normal((k, q - 1))
        u /= np.linalg.norm(u, axis=1, keepdims=True)
        a, be, case = rng.uniform(0.5, 1.5, k), rng.uniform(0.5, 1.5, k), np.arange(k) % 3
        a, be = np.where(case != 1, a, 0.0), np.where(case != 0, be, 0.0)
        s[o:o + k * q] = np.concatenate([a[:, None] * u, a[:, None]], 1).ravel()
        y[o:o + k * q] = np.concatenate([-be[:, None] * u, be[:, None]], 1).ravel()
        o += k * q
    for d in psd:
        V, _ = np.linalg.qr(rng.standard_normal((d, d)))
        lam = np.where(np.arange(d) < d // 2, 1.0, -1.0) * rng.uniform(0.5, 2.0, d)
        k = d * (d + 1) // 2
        s[o:o + k] = _svec((V * np.maximum(lam, 0)) @ V.T)
        y[o:o + k] = _svec((V * np.maximum(-lam, 0)) @ V.T)
        o += k
    b = np.bincount(rows, weights=A.data * x[A.indices], minlength=m) + s
    c = -np.bincount(A.indices, weights=A.data * y[rows], minlength=n)
    return b, c


def _svec_map(d):
    """Position of (i, j), i >= j, in the column-by-column lower triangle, as row and column indices."""
    j, i = np.triu_indices(d)
    return i, j


def _svec(X):
    i, j = _svec_map(X.shape[0])
    return X[i, j] * np.where(i == j, 1.0, SQRT2)


def _sparse_program(scale, seed):
    """The benchmark's large planted program, scaled: 50 nonzeros a row, half the rows orthant, half SOCs of 50."""
    n = int(round(100_000 * scale))
    l, nq = n, max(1, int(round(2000 * scale)))
    m = l + 50 * nq
    A, rows = _sparse(n, m, 50 * m, seed)
    b, c = _planted(np.random.default_rng(seed), A, rows, l, [50] * nq, [])
    return dict(A=A, b=b, c=c, f=0, l=l, q=[50] * nq, s=[])


def _orders(case):
    """Block orders between the case's two bounds (not from the seed: the sizes belong to the case)."""
    return [int(v) for v in np.random.default_rng(1).integers(case["order_low"], case["order_high"] + 1, case["blocks"])]


def _sdp_program(case, seed):
    """The benchmark's planted SDP: PSD blocks and about a hundred orthant rows a block, two entries a row in all."""
    psd = _orders(case)
    l = 98 * len(psd)
    n = 39 * len(psd)
    m = l + sum(d * (d + 1) // 2 for d in psd)
    A, rows = _sparse(n, m, m, seed)
    b, c = _planted(np.random.default_rng(seed), A, rows, l, [], psd)
    return dict(A=A, b=b, c=c, f=0, l=l, q=[], s=psd)


def _lasso_design(case, seed):
    rng = np.random.default_rng(seed)
    p, k = case["rows"], case["cols"]
    F = rng.standard_normal((p, k)) / math.sqrt(p)
    if case["density"] < 1:
        F *= np.random.default_rng(3).random((p, k)) < case["density"]  # the pattern belongs to the case
    return F


def _lasso_rhs(F, rng):
    k = F.shape[1]
    x = np.zeros(k)
    x[rng.choice(k, max(1, k // 20), replace=False)] = rng.standard_normal(max(1, k // 20))
    return F @ x + 0.01 * rng.standard_normal(F.shape[0])


def _portfolios(case, seed):
    """Long-only mean-risk portfolios, k assets and k // 10 factors each (the rows of workloads.portfolio)."""
    sizes = np.random.default_rng(2).integers(case["low"], case["high"] + 1, case["count"])
    rng, out = np.random.default_rng(seed), []
    for k in (int(v) for v in sizes):
        r = max(1, k // 10)
        F, w = rng.standard_normal((r, k)) / math.sqrt(k), np.arange(k, dtype=np.int32)
        counts = np.concatenate([[k], np.ones(k), np.full(r, k), np.ones(k + 1)]).astype(np.int64)
        A = Csr((2 * k + r + 2, k + 1), np.concatenate([[0], np.cumsum(counts)]),
                np.concatenate([w, w, np.tile(w, r), w, [k]]).astype(np.int32),
                np.concatenate([np.ones(k), -np.ones(k), -F.ravel(), -np.sqrt(rng.uniform(0.01, 0.1, k)), [-1.0]]))
        b = np.zeros(2 * k + r + 2)
        b[0] = 1.0
        out.append(dict(A=A, b=b, c=np.concatenate([-rng.normal(0.05, 0.02, k), [1.0]]), f=1, l=k, q=[r + k + 1],
                        s=[]))
    return out


# ---------------------------------------------------------------------------------------------------------------
# what the program holds, and the calls
# ---------------------------------------------------------------------------------------------------------------
_DIR = {"aa": dict(direction=B.DIR_AA), "rb": dict(direction=B.DIR_RB, c0=0.1), "aa_qr": dict(direction=B.DIR_AA_QR)}


def _ok(rc, h=None):
    if rc != B.SCS_OK:
        raise RuntimeError(B.last_error(h))


def _p(t):
    return C.c_void_p(t.data_ptr())


def _points(case, seed):
    """Successive iterates in an SDP's HSDE space: a point whose blocks have spectra on both sides of zero, and three
    more, each a few percent on."""
    psd = _orders(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    l, n = 98 * len(psd), 39 * len(psd)
    N = n + l + sum(d * (d + 1) // 2 for d in psd) + 1
    v = torch.randn(N, generator=g, device="cuda", dtype=torch.float64)
    v[-1] = 1.0
    out = [v]
    for _ in range(3):
        v = v + 0.03 * torch.randn(N, generator=g, device="cuda", dtype=torch.float64)
        out.append(v)
    return out


def _rhs(case, seed):
    """Right-hand sides of two linear systems in a row."""
    n = int(round(100_000 * case["scale"]))
    N = n + n + 50 * max(1, int(round(2000 * case["scale"]))) + 1
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    r = torch.randn(N, generator=g, device="cuda", dtype=torch.float64)
    return [r, r + torch.randn(N, generator=g, device="cuda", dtype=torch.float64)]


def _net_data(case, seed):
    """Parameters (W1, b1, W2, b2, W3, b3 packed), a batch of inputs and targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    di, h, do, rows = case["d_in"], case["hidden"], case["d_out"], case["rows"]

    def uniform(count, fan):
        return (2 * torch.rand(count, generator=g, device="cuda") - 1) / math.sqrt(fan)

    params = torch.cat([uniform(h * di, di), uniform(h, di), uniform(h * h, h), uniform(h, h), uniform(do * h, h),
                        uniform(do, h)])
    X = torch.randn(rows, di, generator=g, device="cuda")
    Y = torch.randn(rows, do, generator=g, device="cuda")
    return params, X, Y


def prepare(case, seed):
    kind = case["kind"]
    # settings of the sweeps over the paper's families; eps is out of reach of the budget
    loop = dict(mem=10, eps=1e-9, cg_rtol=1e-10, cg_adapt=1e-2, max_iters=case.get("iters", 1))
    if kind in ("lasso", "logreg", "pca"):
        if kind == "lasso":
            F = _lasso_design(case, seed)
            prob = W.lasso(F=F, g=_lasso_rhs(F, np.random.default_rng(seed + 1)))
        elif kind == "logreg":
            prob = W.logreg(seed, p=case["cols"], q=case["rows"], lam=10.0)
            # a loose CG on this family stops on an iterate that its own rounding has reached: solve to the end
            loop.update(linsys_direct=case["direct"], cg_adapt=0.0, cg_rtol=1e-12)
        else:
            prob = W.pca_sdp(seed, d=case["order"], lam=0.1)
            loop["threads"] = 1024
        return dict(kind="solve", work=B.Work(prob, **_DIR[case["direction"]], **loop))
    if kind in ("sparse_solve", "sdp_solve"):
        prob = _sparse_program(case["scale"], seed) if kind == "sparse_solve" else _sdp_program(case, seed)
        return dict(kind="solve", work=B.Work(prob, **_DIR[case["direction"]], **loop))
    if kind in ("portfolio", "lasso_batch"):
        if kind == "portfolio":
            probs = _portfolios(case, seed)
            batch = B.Batch(probs, **_DIR["aa"], **loop, linsys_direct=1, threads=256)
        else:
            F = _lasso_design(case, seed)
            prob = W.lasso(F=F, g=_lasso_rhs(F, np.random.default_rng(seed)))
            bcs = [W.lasso_family_bc(F, _lasso_rhs(F, np.random.default_rng([seed, i]))) for i in range(case["count"])]
            batch = B.Batch(shared=(prob, [v[0] for v in bcs], [v[1] for v in bcs]), **_DIR["rb"], **loop,
                            threads=256)
        # results of all instances one after another, as the caller wants them
        out, ptr = [], []
        for rows in ([k.n for k in batch.keeps], [k.m for k in batch.keeps], [k.m for k in batch.keeps]):
            buf = np.empty(sum(rows))
            first = np.concatenate([[0], np.cumsum(rows)[:-1]])
            out.append(buf)
            ptr.append((C.c_void_p * len(rows))(*[buf.ctypes.data + 8 * int(o) for o in first]))
        return dict(kind="batch", batch=batch, out=out, ptr=ptr)
    if kind == "linsys":
        mixed = case["precision"] == "mixed"
        work = B.Work(_sparse_program(case["scale"], seed), cg_rtol=1e-13,
                      precision=B.MIXED if mixed else B.FP64)
        r = _rhs(case, seed)
        return dict(kind=kind, work=work, r=r, out=[torch.empty_like(v) for v in r], slot=2 if mixed else 0)
    if kind == "cone":
        mixed = case["precision"] == "mixed"
        work = B.Work(_sdp_program(case, seed), precision=B.MIXED if mixed else B.FP64)
        v = _points(case, seed)
        return dict(kind=kind, work=work, v=v, out=[torch.empty_like(x) for x in v],
                    precision=B.MIXED if mixed else B.FP64)
    params, X, Y = _net_data(case, seed)
    net = B.MLP(case["d_in"], case["hidden"], case["d_out"], max_batch=case["rows"])
    _ok(B.lib().scs_mlp_set_params(net.h, _p(params)))
    return dict(kind=kind, net=net, X=X, Y=Y, params=params, out=torch.empty_like(Y))


def run(state):
    kind = state["kind"]
    if kind == "solve":
        # the solution as far as it got (NaN while tau is 0) and the iterate that the next call can go on from
        x, y, s, _ = state["work"].solve()
        return {"x": x, "y": y, "s": s, "u": state["work"].get_u()}
    if kind == "batch":
        x, y, s = state["ptr"]
        _ok(B.lib().scs_batch_solve(state["batch"].h, x, y, s, None))
        return dict(zip("xys", state["out"]))
    if kind == "linsys":
        h = state["work"].h
        for r, out in zip(state["r"], state["out"]):
            _ok(B.lib().scs_linsys(h, _p(r), _p(out), state["slot"]), h)
        return state["out"]
    if kind == "cone":
        h = state["work"].h
        for v, out in zip(state["v"], state["out"]):
            _ok(B.lib().scs_project_cone_prec(h, state["precision"], _p(v), _p(out), None), h)
        return [o.float() if state["precision"] == B.MIXED else o for o in state["out"]]
    net = state["net"]
    if kind == "mlp_forward":
        return net.forward(state["X"], state["out"])
    loss = net.train_step(state["X"], state["Y"], 1e-4)
    _ok(B.lib().scs_mlp_get_params(net.h, _p(state["params"])))
    return {"loss": np.float32(loss), "params": state["params"]}


# ---------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------
def _size(case):
    """n, m and nonzeros of a case's problem."""
    kind = case["kind"]
    if kind in ("lasso", "lasso_batch"):
        p, k = case["rows"], case["cols"]
        return 2 * k + 1, 2 * k + p + 2, 4 * k + 2 + int(p * k * case["density"])
    if kind == "logreg":
        q, p = case["rows"], case["cols"]
        return 2 * p + 3 * q, 2 * p + 7 * q, 4 * p + 6 * q + p * q
    if kind == "pca":
        k = case["order"] * (case["order"] + 1) // 2
        return 2 * k, 1 + 3 * k, 5 * k + case["order"]
    if kind in ("linsys", "sparse_solve"):
        n = int(round(100_000 * case["scale"]))
        m = n + 50 * max(1, int(round(2000 * case["scale"])))
        return n, m, 50 * m
    psd = _orders(case)
    m = 98 * len(psd) + sum(d * (d + 1) // 2 for d in psd)
    return 39 * len(psd), m, m


def work(case):
    """Data read once, results written once; the products with A and A^T that the iterations need at the least (one
    pair to test for termination, and for each linear system one pair and one product), and about 9 d^3 for a
    symmetric eigendecomposition and the product that rebuilds the projection."""
    kind = case["kind"]
    if kind in ("mlp_train", "mlp_forward"):
        di, h, do, rows = case["d_in"], case["hidden"], case["d_out"], case["rows"]
        weights, params = h * di + h * h + do * h, h * di + h * h + do * h + 2 * h + do
        if kind == "mlp_forward":
            return {"bytes": 2 * weights + 4 * rows * (di + do), "flops": 2 * rows * weights}
        # parameters and both moments read and written, gradients and the GEMMs' BF16 copies written, both copied out
        return {"bytes": (6 * 4 + 2 * 2 + 4 + 2 * 4) * params + 4 * rows * (di + do), "flops": 6 * rows * weights}
    if kind == "portfolio":
        sizes = np.random.default_rng(2).integers(case["low"], case["high"] + 1, case["count"]).astype(np.int64)
        nnz = sizes * (sizes // 10 + 3)
        return {"bytes": int((12 * nnz + 8 * 8 * sizes).sum()),
                "flops": int(case["iters"] * (2 * sizes * sizes + 10 * nnz).sum())}
    n, m, nnz = _size(case)
    data = 12 * nnz + 8 * (n + m)
    if kind == "linsys":
        esize = 8 if case["precision"] == "mixed" else 12
        # two systems; conjugate gradients needs some tens of products with each of A and A^T for 13 digits
        return {"bytes": 2 * (30 * 2 * esize * nnz + 16 * (n + m)), "flops": 2 * 30 * 4 * nnz}
    eig = sum(9 * d ** 3 for d in (_orders(case) if "order_low" in case else [case.get("order", 0)]))
    if kind == "cone":
        return {"bytes": 4 * 16 * (n + m), "flops": 4 * eig}
    count, its = case.get("count", 1), case["iters"]
    return {"bytes": data + count * 8 * (2 * n + 3 * m), "flops": count * its * (10 * nnz + eig)}


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------------------------
def _exact_linsys(case, seed):
    """(I + Q)^{-1} r by conjugate gradients on I + A^T A, to the last digits that 64 bits give."""
    prob = _sparse_program(case["scale"], seed)
    A = prob["A"]
    m, n = A.shape
    col = torch.as_tensor(A.indices, device="cuda").long()
    row = torch.repeat_interleave(torch.arange(m, device="cuda"), torch.as_tensor(np.diff(A.indptr), device="cuda"))
    val = torch.as_tensor(A.data, device="cuda")
    M = torch.sparse_coo_tensor(torch.stack([row, col]), val, (m, n)).to_sparse_csr()
    Mt = torch.sparse_coo_tensor(torch.stack([col, row]), val, (n, m)).coalesce().to_sparse_csr()

    def solve(a, e):
        rhs = a - Mt @ e
        x = torch.zeros_like(rhs)
        for _ in range(2):  # restarted once from the true residual
            r = rhs - x - Mt @ (M @ x)
            p, rr = r.clone(), torch.dot(r, r)
            for _ in range(400):
                if float(rr) <= 1e-30 * float(torch.dot(rhs, rhs)):
                    break
                q = p + Mt @ (M @ p)
                al = rr / torch.dot(p, q)
                x += al * p
                r -= al * q
                new = torch.dot(r, r)
                p, rr = r + (new / rr) * p, new
        return torch.cat([x, e + M @ x])

    h = torch.as_tensor(np.concatenate([prob["c"], prob["b"]]), device="cuda")
    g = solve(h[:n], h[n:])
    out = []
    for r in _rhs(case, seed):
        z = solve(r[:n], r[n:-1])
        tau = (r[-1] + torch.dot(h, z)) / (1 + torch.dot(h, g))
        out.append(torch.cat([z - tau * g, tau.reshape(1)]))
    return out


def _exact_cone(case, seed):
    """Each block of psi projected by a 64-bit eigendecomposition (the dual cone of a PSD block is itself)."""
    psd = _orders(case)
    n, l = 39 * len(psd), 98 * len(psd)
    out = []
    for v in _points(case, seed):
        if case["precision"] == "mixed":
            v = v.float().double()
        u = v.clone()
        u[n:n + l].clamp_(min=0)
        u[-1].clamp_(min=0)
        o = n + l
        first = {}
        for d in psd:
            first.setdefault(d, []).append(o)
            o += d * (d + 1) // 2
        for d, offs in first.items():
            i, j = (torch.as_tensor(t, device="cuda") for t in _svec_map(d))
            at = torch.as_tensor(offs, device="cuda")[:, None] + torch.arange(len(i), device="cuda")
            scale = torch.where(i == j, 1.0, SQRT2).double()
            X = torch.zeros(len(offs), d, d, dtype=torch.float64, device="cuda")
            X[:, i, j] = v[at] / scale
            lam, V = torch.linalg.eigh(X)  # reads the lower triangle
            X = (V * lam.clamp(min=0)[:, None, :]) @ V.transpose(1, 2)
            u[at] = X[:, i, j] * scale
        out.append(u)
    return out


def _exact_net(case, seed):
    params, X, Y = (t.double() for t in _net_data(case, seed))
    di, h, do = case["d_in"], case["hidden"], case["d_out"]
    split = torch.split(params, [h * di, h, h * h, h, do * h, do])
    W1, b1, W2, b2, W3, b3 = split[0].view(h, di), split[1], split[2].view(h, h), split[3], split[4].view(do, h), split[5]
    h1 = torch.relu(X @ W1.T + b1)
    h2 = torch.relu(h1 @ W2.T + b2)
    y = h2 @ W3.T + b3
    if case["kind"] == "mlp_forward":
        return y
    dy = (y - Y) / Y.numel()
    d2 = (dy @ W3) * (h2 > 0)
    d1 = (d2 @ W2) * (h1 > 0)
    g = torch.cat([(d1.T @ X).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), (dy.T @ h2).reshape(-1),
                   dy.sum(0)])
    # the first step of Adam: the bias corrections cancel the decay rates
    return {"loss": 0.5 * ((y - Y) ** 2).mean(), "params": params - 1e-4 * g / (g.abs() + 1e-8)}


def exact(case, seed):
    """None for the solves: the iterate after a given number of iterations has no value but the algorithm's own."""
    if case["kind"] == "linsys":
        return _exact_linsys(case, seed)
    if case["kind"] == "cone":
        return _exact_cone(case, seed)
    if case["kind"].startswith("mlp"):
        return _exact_net(case, seed)
    return None
