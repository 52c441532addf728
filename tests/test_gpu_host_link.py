"""ax_local_host on page-locked float32 buffers (the kernel reads and writes them
over the host link, in whole lines through shared memory) against ax_local on
the device: the same operations in the same order, so the same bits, for every
order and kind, with counts of elements that leave the last block ragged and
buffers that start at any word; and nothing is written beyond the last element."""
import numpy as np
import pytest

from paper_2504_07042_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ax():
    from paper_2504_07042_gb300 import build

    build.build()
    from paper_2504_07042_gb300 import ax as _ax

    return _ax


@pytest.mark.parametrize("kind", ["trilinear", "stored", "parallelepiped", "partial"])
@pytest.mark.parametrize("N", range(1, 16))
def test_same_bits_as_on_the_device(ax, kind, N):
    for (ex, ey, ez), shift in (((1, 1, 1), 0), ((5, 3, 3), 1), ((7, 5, 2), 3)):
        V = inputs.parallelepiped_vertices(ex, ey, ez) if kind == "parallelepiped" else \
            inputs.box_vertices(ex, ey, ez, perturb=0.1, seed=2)
        op = ax.Ax(torch.from_numpy(V).to(DEV), N, kind, "fp32")
        n = op.E * op.n3
        Xb = torch.from_numpy(np.random.default_rng(N).uniform(-1, 1, n + shift).astype(np.float32)).pin_memory()
        Yb = torch.full((n + shift + 4,), 7.0).pin_memory()
        X = Xb[shift:].to(DEV)
        ref = op.ax_local(X, torch.empty_like(X)).cpu()
        op.ax_local_host(Xb[shift:], Yb[shift:])
        assert torch.equal(Yb[shift:shift + n], ref)
        assert (Yb[shift + n:] == 7.0).all() and (Yb[:shift] == 7.0).all()
