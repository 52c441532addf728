"""Gradients of a batch after a larger one on the same network: the partial sums
of the split batch, the column sums and the squares lie in buffers that the
larger batch left full, at other strides and with fewer splits.  Every layer's
gradients against the FP64 oracle, with the tolerance of test_gpu_mlp.py (8 bf16
roundings of every entry's own error scale), and the bits of a fresh network."""
import numpy as np
import pytest

from test_gpu_mlp import I, U_BF16, _scales, _setup, _split

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ax():
    from paper_2504_07042_gb300 import build

    build.build()
    from paper_2504_07042_gb300 import ax as _ax

    return _ax


@pytest.mark.parametrize("large,small", [(4128, 32), (1024, 352), (352, 96)])
def test_gradients_after_a_larger_batch(ax, large, small):
    from oracle import mlp as om

    mlp, Xd, Td, Xq, T, Pq = _setup(ax, seed=23, M=large)
    mlp.ax_mlp_grad(Xd, Td)
    Xs, Ts = Xd[:small].contiguous(), Td[:small].contiguous()
    loss, g = mlp.ax_mlp_grad(Xs, Ts)
    fresh = _setup(ax, seed=23, M=large)[0]
    loss_ref, g_ref = fresh.ax_mlp_grad(Xs, Ts)
    assert loss == loss_ref and np.array_equal(g, g_ref)
    L, gref = om.grads(Pq, Xq[:small], T[:small])
    assert abs(loss - L) / L < 1e-2
    G = _split(g.astype(np.float64))
    assert np.all(G[0][:, I:] == 0.0)
    G[0] = G[0][:, :I]
    _, scales = _scales(Pq, Xq[:small], T[:small])
    for name, a, b, sc in zip(("dW1", "db1", "dW2", "db2", "dW3", "db3"), G, gref, scales):
        assert (np.abs(a - b) / (U_BF16 * sc)).max() < 8.0, name
