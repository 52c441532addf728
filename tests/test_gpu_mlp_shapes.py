"""The network's GEMMs at the edges of their tiles, against the FP64 oracle:
row counts around the 128-row tile, and for the gradients batches that do not
fill a 64-row contraction block, leave ragged splits of the batch between the
CTAs or exceed one wave; targets and outputs that are not 16-byte aligned.

Tolerances are those of test_gpu_mlp.py (8 bf16 roundings of every entry's
own error scale), which do not depend on the batch."""
import numpy as np
import pytest

from test_gpu_mlp import DEV, I, O, U_BF16, _scales, _setup, _split, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ax():
    from paper_2504_07042_gb300 import build

    build.build()
    from paper_2504_07042_gb300 import ax as _ax

    return _ax


@pytest.mark.parametrize("M", [1, 31, 128, 129, 1000])
@pytest.mark.parametrize("shift", [0, 1])
def test_forward_rows(ax, M, shift):
    from oracle import mlp as om

    mlp, Xd, _, Xq, _, Pq = _setup(ax, seed=21, M=M)
    buf = torch.full((M * O + 8,), float("nan"), dtype=torch.float32, device=DEV)
    Y = buf[shift:shift + M * O].view(M, O)
    mlp.ax_mlp_forward(Xd, Y)
    Yref, _ = om.forward(Pq, Xq)
    Ys, _ = _scales(Pq, Xq, np.zeros_like(Yref))
    assert (np.abs(Y.cpu().numpy() - Yref) / (U_BF16 * Ys)).max() < 8.0
    # nothing written beyond the rows asked for
    assert torch.isnan(buf[shift + M * O:]).all() and torch.isnan(buf[:shift]).all()


@pytest.mark.parametrize("M,shift", [(32, 0), (96, 0), (160, 1), (352, 0), (4128, 0)])
def test_gradient_batches(ax, M, shift):
    from oracle import mlp as om

    mlp, Xd, Td, Xq, T, Pq = _setup(ax, seed=22, M=M)
    buf = torch.empty(M * O + 4, dtype=torch.float32, device=DEV)
    Ts = buf[shift:shift + M * O].view(M, O)
    Ts.copy_(Td)
    loss, g = mlp.ax_mlp_grad(Xd, Ts)
    Lref, gref = om.grads(Pq, Xq, T)
    assert abs(loss - Lref) / Lref < 1e-2
    G = _split(g.astype(np.float64))
    assert np.all(G[0][:, I:] == 0.0)
    G[0] = G[0][:, :I]
    _, scales = _scales(Pq, Xq, T)
    for name, a, b, sc in zip(("dW1", "db1", "dW2", "db2", "dW3", "db3"), G, gref, scales):
        assert (np.abs(a - b) / (U_BF16 * sc)).max() < 8.0, name
    # a second batch of another size on the same network reuses the buffers
    loss2, g2 = mlp.ax_mlp_grad(Xd[:32].contiguous(), Ts[:32].contiguous())
    Lref2, gref2 = om.grads(Pq, Xq[:32], T[:32])
    assert abs(loss2 - Lref2) / Lref2 < 1e-2
