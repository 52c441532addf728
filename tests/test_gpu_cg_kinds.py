"""The fused CG iteration at the kinds and orders that test_gpu_cg_fused.py leaves
out: parallelepiped and partial elements, the orders in between (each has its own
shape, layout and loads), and the persistent batch with every kind, against the
oracle's operator under CG in float64 after the same number of iterations.

Tolerances as in test_gpu_cg_fused.py: CG magnifies the operator's rounding
errors a little in every step; after at most 7 iterations 1e-9 leaves four
digits over the double-word operator's 1e-13, and 2e-4 over float32's 2e-7."""
import numpy as np
import pytest

from paper_2504_07042_gb300 import inputs
from test_gpu_cg_fused import DEV, _cg, torch

pytestmark = pytest.mark.gpu
TOL = {"f64dw": 1e-9, "fp32": 2e-4}


@pytest.fixture(scope="module")
def ax():
    from paper_2504_07042_gb300 import build

    build.build()
    from paper_2504_07042_gb300 import ax as _ax

    return _ax


def _system(orc, kind, box, N, seed):
    V = inputs.parallelepiped_vertices(*box) if kind == "parallelepiped" else \
        inputs.box_vertices(*box, perturb=0.1, seed=seed)
    G, _ = orc.factors(V, N)
    gid, ng = inputs.box_global_ids(*box, N)
    mask = inputs.box_boundary_mask(*box, N)
    free = (mask == 0).astype(np.float64)

    def A(u):
        return orc.gather(orc.axlocal(G, orc.scatter(u, gid), N), gid, ng) * free

    dg = orc.gather(orc.element_diagonals(G, N), gid, ng)
    inv = np.where(free > 0, 1.0 / np.where(free > 0, dg, 1.0), 0.0)
    rng = np.random.default_rng(100 + seed)
    return V, gid, ng, mask, A, inv, rng.uniform(-1, 1, ng) * free, rng.uniform(-1, 1, ng) * free


def _dev(V, gid, mask):
    return torch.from_numpy(V).to(DEV), torch.from_numpy(gid).to(DEV), torch.from_numpy(mask).to(DEV)


@pytest.mark.parametrize("prec", ["f64dw", "fp32"])
@pytest.mark.parametrize("kind,box,N,iters", [
    ("parallelepiped", (5, 4, 3), 1, 7), ("parallelepiped", (3, 3, 2), 4, 6), ("parallelepiped", (3, 2, 2), 7, 7),
    ("parallelepiped", (2, 2, 1), 11, 5), ("parallelepiped", (2, 1, 1), 15, 4), ("partial", (3, 3, 2), 3, 6),
    ("partial", (3, 2, 2), 7, 6), ("partial", (2, 2, 1), 10, 5), ("trilinear", (3, 3, 3), 3, 7),
    ("trilinear", (3, 2, 1), 8, 6), ("stored", (3, 2, 1), 9, 5), ("trilinear", (2, 2, 1), 12, 5),
    ("stored", (2, 2, 1), 13, 5), ("parallelepiped", (2, 1, 1), 13, 5), ("trilinear", (2, 1, 1), 14, 4)])
def test_iterates(ax, orc, kind, box, N, iters, prec):
    V, gid, ng, mask, A, inv, b, x0 = _system(orc, kind, box, N, seed=5)
    Vd, gd, md = _dev(V, gid, mask)
    op = ax.Ax(Vd, N, kind, prec)
    op.gs_setup(gd, ng, md)
    x = torch.from_numpy(x0).to(DEV, op.dtype)
    it, _, st = op.pcg_solve(torch.from_numpy(b).to(DEV, op.dtype), x, rtol=0.0, maxit=iters)
    assert st == ax.AX_ENOTCONV and it == iters
    ref = _cg(A, b, inv, x0, iters)
    assert np.max(np.abs(x.double().cpu().numpy() - ref)) <= TOL[prec] * np.max(np.abs(ref))


@pytest.mark.parametrize("kind", ["trilinear", "stored", "parallelepiped", "partial"])
def test_persistent_batch_iterates(ax, orc, kind):
    systems = [(box, N) + _system(orc, kind, box, N, seed=s) for s, (box, N) in enumerate(
        [((3, 3, 2), 3), ((4, 3, 3), 1), ((2, 2, 2), 5), ((2, 2, 1), 7), ((3, 2, 1), 8), ((2, 1, 1), 9)])]
    meshes = []
    for box, N, V, gid, ng, mask, *_ in systems:
        Vd, gd, md = _dev(V, gid, mask)
        meshes.append((Vd, N, gd, ng, md))
    bt = ax.AxBatch(meshes, kind, "fp32")
    assert bt.ax_batch_info()["iteration_launches"] == 1
    for iters in (4, 7):
        b = torch.from_numpy(np.concatenate([s[8] for s in systems])).to(DEV, torch.float32)
        x = torch.from_numpy(np.concatenate([s[9] for s in systems])).to(DEV, torch.float32)
        bt.ax_batch_pcg(b, x, rtol=0.0, maxit=iters, graph=1, check=False)
        got = x.double().cpu().numpy()
        for m, (box, N, V, gid, ng, mask, A, inv, bm, x0) in enumerate(systems):
            ref = _cg(A, bm, inv, x0, iters)
            err = np.max(np.abs(got[bt.global_offsets[m]:bt.global_offsets[m + 1]] - ref)) / np.max(np.abs(ref))
            assert err <= TOL["fp32"], (m, N, err)
