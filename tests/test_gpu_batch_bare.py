"""A float32 batch with nodes that no element has keeps its persistent iteration
(a small kernel beside it updates those nodes): it agrees with the launches per
phase, its waits stay bounded by ax_batch_set_wait, and a mesh that Jacobi
cannot solve (such a node without a Dirichlet mask has a zero on the diagonal)
leaves the other meshes alone.

Tolerance: the two paths add float32 sums in another order, which CG magnifies a
little in every step; after 8 iterations 2e-4 leaves three digits over float32's
2e-7."""
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


def _batch(ax, spare, masked):
    """Four meshes, mesh m with spare[m] nodes beyond those of its elements."""
    out = []
    for s, (ex, ey, ez, N) in enumerate([(3, 2, 2, 3), (4, 4, 3, 5), (2, 2, 2, 7), (2, 1, 1, 9)]):
        V = inputs.box_vertices(ex, ey, ez, perturb=0.1, seed=s)
        gid, ng = inputs.box_global_ids(ex, ey, ez, N)
        mask = np.concatenate([inputs.box_boundary_mask(ex, ey, ez, N), np.full(spare[s], masked, np.uint8)])
        out.append((torch.from_numpy(V).to(DEV), N, torch.from_numpy(gid).to(DEV), ng + spare[s],
                    torch.from_numpy(mask).to(DEV)))
    return ax.AxBatch(out, "trilinear", "fp32")


def _solve(bt, seed):
    rng = np.random.default_rng(seed)
    b = torch.from_numpy(rng.uniform(0.5, 1.5, bt.n_global)).to(DEV, torch.float32)
    x = torch.from_numpy(rng.uniform(-1, 1, bt.n_global)).to(DEV, torch.float32)
    st = bt.ax_batch_pcg(b, x, rtol=0.0, maxit=8, graph=1, check=False)[2]
    return x.double().cpu().numpy(), st


@pytest.mark.parametrize("spare,masked", [((1, 0, 0, 0), 1), ((0, 3000, 1, 300), 1), ((0, 2, 0, 0), 0)])
def test_agrees_with_the_launches_per_phase(ax, spare, masked):
    bt = _batch(ax, spare, masked)
    assert bt.ax_batch_info() == {"persistent": 1, "local_launches": 1, "iteration_launches": 2}
    x, _ = _solve(bt, 3)
    bt.ax_batch_set_persistent(False)
    ref, _ = _solve(bt, 3)
    for m in range(bt.B):
        a, b = bt.global_offsets[m], bt.global_offsets[m + 1]
        if spare[m] and not masked:
            assert not np.isfinite(ref[a:b]).any() and not np.isfinite(x[a:b]).any()
        else:
            assert np.max(np.abs(x[a:b] - ref[a:b])) <= 2e-4 * np.max(np.abs(ref[a:b]))


def test_waits_stay_bounded(ax):
    bt = _batch(ax, (0, 1, 0, 0), 1)
    bt.ax_batch_set_wait(1_000_000, stuck_mesh=2)
    assert _solve(bt, 5)[1] == ax.AX_ETIMEOUT
    bt.ax_batch_set_wait(2_000_000_000, stuck_mesh=-1)
    x, st = _solve(bt, 5)
    assert st == ax.AX_ENOTCONV and np.isfinite(x).all()
