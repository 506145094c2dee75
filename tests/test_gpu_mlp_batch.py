"""The training pass at batches of one and of several pieces, with whole and
short last ones (a piece is 512 rows up to 16,384 rows, 1/32 of the batch
above): layer by layer against the reference, with the bounds of
test_gpu_mlp_layers; beyond what a trace takes, against the gradient of a block that the
batch repeats (2/B is a power of two: only the order of the sums differs)."""
import numpy as np
import pytest

from paper_1401_1757_gb300 import rsv
from test_gpu_mlp_layers import U32, backward_report, ctx, params  # noqa: F401

pytestmark = pytest.mark.gpu


def batch(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.normal(0, 1, (n, 32)).astype(np.float32)
    X[:, 20:] = 0.0
    return X, rng.normal(0, 1, n).astype(np.float32)


@pytest.mark.parametrize("n", [128, 512, 640, 1152, 4096])
def test_backward_by_pieces(ctx, n):  # noqa: F811
    p = params(31)
    X, t = batch(n, n)
    rsv.rsv_mlp_set_params(ctx, p)
    tr = rsv.rsv_mlp_trace(ctx, X, backend=rsv.RSV_MLP_MMA_SYNC, target=t)
    bw = backward_report(p, tr, t.astype(np.float64))
    assert max(bw.values()) <= 1.0, bw
    g, loss = rsv.rsv_mlp_gradient(ctx, X, t)
    assert np.array_equal(g.astype(np.float64), tr["grads"])
    sq = (tr["y"] - t) ** 2
    assert abs(loss - sq.mean()) <= (n + 3) * U32 * sq.mean()


@pytest.mark.parametrize("n", [16384, 32768])
def test_repeated_block(ctx, n):  # noqa: F811
    p = params(32)
    X, t = batch(512, 7)
    rsv.rsv_mlp_set_params(ctx, p)
    tr = rsv.rsv_mlp_trace(ctx, X, backend=rsv.RSV_MLP_MMA_SYNC, target=t)
    g, loss = rsv.rsv_mlp_gradient(ctx, np.tile(X, (n // 512, 1)), np.tile(t, n // 512))
    # sums of |terms|: |A|^T |dZ| a weight, |dZ| a bias; the largest bounds a layer's
    ref, o = tr["grads"], 0
    for l, k in enumerate((32, 256, 256, 256)):
        A = tr["Xb"] if l == 0 else tr["A"][l - 1]
        w = np.abs(A).T @ np.abs(tr["dZ"][l])
        bound = np.concatenate([(w[:32] + w[32:] if l == 0 else w).ravel(), np.abs(tr["dZ"][l]).sum(0)])
        e = np.abs(g[o:o + bound.size] - ref[o:o + bound.size])
        assert np.all(e <= 2 * (n + 3) * U32 * bound + 1e-30), l
        o += bound.size
    assert abs(loss - ((tr["y"] - t) ** 2).mean()) <= 2 * (n + 3) * U32 * loss
