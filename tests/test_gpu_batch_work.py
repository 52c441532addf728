"""The work that a batch keeps between solves (vectors, captured iterations,
inverted diagonal): solves with other buffers, other counts, the other path and
after tuning, in one batch, against a fresh batch for each; and a batch with
nodes that no element has, which takes the launches per group.

Tolerance: the same path sums in the same order, so the results are the same
bits.  Another path or tiling changes the order of float32 sums; CG magnifies
that a little in every step: after at most 9 iterations 2e-4 leaves three digits
over float32's 2e-7."""
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


def _meshes(spare=0):
    out = []
    for s, (ex, ey, ez, N) in enumerate([(3, 2, 2, 3), (2, 2, 1, 5), (2, 2, 2, 7), (2, 1, 1, 9)]):
        V = inputs.box_vertices(ex, ey, ez, perturb=0.1, seed=s)
        gid, ng = inputs.box_global_ids(ex, ey, ez, N)
        mask = np.concatenate([inputs.box_boundary_mask(ex, ey, ez, N), np.ones(spare, np.uint8)])
        out.append((torch.from_numpy(V).to(DEV), N, torch.from_numpy(gid).to(DEV), ng + spare,
                    torch.from_numpy(mask).to(DEV)))
    return out


def _solve(bt, seed, iters):
    """x after `iters` iterations from a start that is not zero, in new buffers."""
    rng = np.random.default_rng(seed)
    b = torch.from_numpy(rng.uniform(0.5, 1.5, bt.n_global)).to(DEV, bt.dtype)
    x = torch.from_numpy(rng.uniform(-1, 1, bt.n_global)).to(DEV, bt.dtype)
    bt.ax_batch_pcg(b, x, rtol=0.0, maxit=iters, graph=1, check=False)
    return x.double().cpu().numpy()


def _close(x, ref):
    return np.max(np.abs(x - ref)) <= 2e-4 * np.max(np.abs(ref))


@pytest.mark.parametrize("prec", ["fp32", "f64dw"])
def test_kept_work_changes_nothing(ax, prec):
    bt = ax.AxBatch(_meshes(), "trilinear", prec)
    for seed, iters in [(1, 9), (2, 4), (3, 1), (1, 9)]:
        assert np.array_equal(_solve(bt, seed, iters), _solve(ax.AxBatch(_meshes(), "trilinear", prec), seed, iters))
    if prec == "fp32":
        ref = _solve(bt, 4, 7)
        for on in (False, True):
            bt.ax_batch_set_persistent(on)
            x = _solve(bt, 4, 7)
            assert _close(x, ref)
        assert np.array_equal(x, ref)
        bt.ax_batch_tune()
        assert _close(_solve(bt, 4, 7), ref)


def test_nodes_without_an_element(ax):
    spare = 5
    bt, loose = ax.AxBatch(_meshes(), "trilinear", "fp32"), ax.AxBatch(_meshes(spare), "trilinear", "fp32")
    assert bt.ax_batch_info()["iteration_launches"] == 1 and loose.ax_batch_info()["iteration_launches"] > 1
    rng = np.random.default_rng(9)
    b = rng.uniform(0.5, 1.5, bt.n_global)
    lo, hi = bt.global_offsets, loose.global_offsets
    bl = np.ones(loose.n_global)
    for m in range(bt.B):
        bl[hi[m]:hi[m] + lo[m + 1] - lo[m]] = b[lo[m]:lo[m + 1]]
    out = []
    for q, v in ((bt, b), (loose, bl)):
        x = torch.zeros(q.n_global, dtype=torch.float32, device=DEV)
        q.ax_batch_pcg(torch.from_numpy(v).to(DEV, torch.float32), x, rtol=0.0, maxit=8, graph=1, check=False)
        out.append(x.double().cpu().numpy())
    same = np.concatenate([out[1][hi[m]:hi[m] + lo[m + 1] - lo[m]] for m in range(bt.B)])
    assert _close(same, out[0])
