"""A batched solve whose bounded wait runs out: the caller's x keeps the initial
guess, bit for bit and on the Dirichlet nodes too (a mesh can stand between the
two halves of an iteration then, and what it holds is no iterate of CG), and
the batch solves normally afterwards.  The wait runs out in the first iteration
(a dependency that nothing completes) or, with a budget of a nanosecond, in any
one in which an item is not ready at once."""
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


@pytest.mark.parametrize("budget,stuck", [(1_000_000, 1), (1, -1)])
def test_x_keeps_the_initial_guess(ax, budget, stuck):
    meshes = []
    for s, (ex, ey, ez, N) in enumerate([(4, 4, 3, 3), (3, 3, 3, 5), (3, 2, 2, 7)]):
        gid, ng = inputs.box_global_ids(ex, ey, ez, N)
        meshes.append((torch.from_numpy(inputs.box_vertices(ex, ey, ez, perturb=0.1, seed=s)).to(DEV), N,
                       torch.from_numpy(gid).to(DEV), ng,
                       torch.from_numpy(inputs.box_boundary_mask(ex, ey, ez, N)).to(DEV)))
    bt = ax.AxBatch(meshes, "trilinear", "fp32")
    rng = np.random.default_rng(6)
    b = torch.from_numpy(rng.uniform(0.5, 1.5, bt.n_global)).to(DEV, torch.float32)
    x0 = torch.from_numpy(rng.uniform(0.5, 1.5, bt.n_global)).to(DEV, torch.float32)
    ref = x0.clone()
    bt.ax_batch_pcg(b, ref, rtol=0.0, maxit=12, check=False)
    bt.ax_batch_set_wait(budget, stuck)
    for _ in range(5):
        x = x0.clone()
        _, _, st = bt.ax_batch_pcg(b, x, rtol=0.0, maxit=12, check=False)
        assert st == ax.AX_ETIMEOUT or stuck < 0
        assert torch.equal(x, x0 if st == ax.AX_ETIMEOUT else ref)
    bt.ax_batch_set_wait(2_000_000_000, -1)
    x = x0.clone()
    bt.ax_batch_pcg(b, x, rtol=0.0, maxit=12, check=False)
    assert torch.equal(x, ref)
