"""Loss and gradient of the branching network over node sizes at the edges of
the kernels' tiles (16 rows, 8 warps per block, 1 to 8 blocks per node), nodes
that take no part (not closed, one row, no targets), and feature rows that are
only 2-byte aligned, against the FP64 reference. Scores likewise."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp_ref as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def libs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_21552_gb300 import build
    build.build()
    from paper_2601_21552_gb300 import api, binding
    return api, binding


def _bits(a):
    f = np.asarray(a, np.float32).view(np.uint32).astype(np.uint64)
    return ((f + 0x7FFF + ((f >> 16) & 1)) >> 16).astype(np.uint16)


SIZES = {
    "one": [300],
    "edges": [1, 2, 15, 16, 17, 31, 32, 33, 127, 128, 129, 255, 257],
    "one_large": [40007],
    "split8": [129] * 38,
    "split4": [257, 1, 64] * 13,
    "split2": [65, 130] * 40,
    "strided": [17, 40, 3] * 120,
}


@pytest.mark.parametrize("offset", [0, 1, 2], ids=["aligned", "off1", "off2"])
@pytest.mark.parametrize("sizes", SIZES.values(), ids=SIZES.keys())
def test_gradient_matches_fp64_at_tile_edges(libs, sizes, offset):
    api, B = libs
    rng = np.random.default_rng(len(sizes))
    n, rows = len(sizes), sum(sizes)
    xb = _bits(rng.normal(size=(rows, 16)))
    target = rng.integers(0, 6, rows).astype(np.float32)
    begin = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.int64)
    closed = np.ones(n, np.int32)
    if n > 4:
        closed[3] = 0
        target[begin[4]:begin[4] + sizes[4]] = 0
    buf = torch.zeros(rows * 16 + 8, dtype=torch.int16, device="cuda")
    buf[offset:offset + rows * 16] = torch.from_numpy(xb.view(np.int16).reshape(-1)).cuda()
    tr = api.Trace(4, n, rows)
    tr.target.copy_(torch.from_numpy(target))
    tr.node_row.copy_(torch.from_numpy(begin))
    tr.node_nrows.copy_(torch.tensor(sizes, dtype=torch.int32))
    tr.node_closed.copy_(torch.from_numpy(closed))
    t = tr.struct()
    t.x = buf.data_ptr() + 2 * offset
    net = api.Mlp(seed=11)
    s = torch.cuda.current_stream().cuda_stream
    grad = torch.full((R.NPARAM + 2,), 7.0, device="cuda")
    ds = torch.full((rows + 1,), 9.0, device="cuda")
    assert B._lib.scuba_mlp_grad(ctypes.byref(t), 0, n, net.weights.data_ptr(), grad.data_ptr(),
                                 ds.data_ptr(), s) == 0
    scores = torch.full((rows + 1,), 5.0, device="cuda")
    assert B._lib.scuba_mlp_forward(t.x, rows, net.weights.data_ptr(), scores.data_ptr(), s) == 0
    W1, b1, w2, b2 = R.unpack_weights(net.weights.cpu().numpy())
    X = R.bf16_to_f64(xb)
    tgt = target.astype(np.float64)
    nodes = [(int(b), m) for b, m, c in zip(begin, sizes, closed) if c]
    p = R.flat(W1, b1, w2, b2)
    sc = R.scores(X, W1, b1, w2, b2)
    want_ds = np.zeros(rows)
    used = 0
    for b, m in nodes:
        ts = tgt[b:b + m].sum()
        if m > 1 and ts > 0:
            e = np.exp(sc[b:b + m] - sc[b:b + m].max())
            want_ds[b:b + m] = e / e.sum() - tgt[b:b + m] / ts
            used += 1
    g = grad.cpu().numpy().astype(np.float64)
    # 1,024 FP32 sums of BF16 products: 1e-5 is 80 units in the last place
    assert np.abs(scores.cpu().numpy()[:rows] - sc).max() <= 1e-5 * max(1.0, np.abs(sc).max())
    assert scores[rows].item() == 5.0 and ds[rows].item() == 9.0
    assert np.abs(ds.cpu().numpy()[:rows] - want_ds).max() <= 2e-5
    assert g[R.NPARAM + 1] == used
    want_loss = R.loss(p, X, nodes, tgt)
    assert abs(g[R.NPARAM] - want_loss) <= 1e-4 * max(1.0, abs(want_loss))
    want = R.grad(p, X, nodes, tgt)
    # dH is rounded to BF16 (2^-9 relative) before dW1; the rest is FP32
    bound = 2.0 ** -9 * (np.abs(X).T @ (np.abs(np.outer(want_ds, w2)))).reshape(-1)
    assert (np.abs(g[:1024] - want[:1024]) <= bound + 2e-5 * max(1, used)).all()
    assert np.abs(g[1024:R.NPARAM] - want[1024:]).max() <= 2e-4 * max(1.0, np.abs(want).max())
