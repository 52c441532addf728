"""The fused CG iteration (FP32 and double-word contexts: the direction, the
update of x and p.w inside AxLocal, gather and update in one kernel) against
the oracle's CG after the same number of iterations, where its bookkeeping can
go wrong: odd and even counts (the direction changes buffers), counts below,
at and past one captured block of 16, no preconditioner, a start that is not
zero, one element, orders whose CTA holds several elements with a ragged last
one; and a numbering with nodes that no element has, which takes the general
iteration.

Tolerance: CG's iterates magnify the operator's rounding errors a little in
every step; after at most 20 iterations on these meshes (condition below 1e3)
1e-9 leaves four digits over the double-word operator's 1e-13, and 2e-4 over
float32's 2e-7 likewise."""
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


def _cg(A, b, inv, x, iters):
    """Plain preconditioned CG in float64 (A: the assembled operator)."""
    r = b - A(x)
    z = inv * r
    p, rz = z.copy(), r @ z
    for _ in range(iters):
        w = A(p)
        alpha = rz / (p @ w)
        x = x + alpha * p
        r = r - alpha * w
        z = inv * r
        rz, old = r @ z, rz
        p = z + (rz / old) * p
    return x


def _problem(orc, box, N, extra=0):
    V = inputs.box_vertices(*box, perturb=0.1, seed=5)
    G, _ = orc.factors(V, N)
    gid, ng = inputs.box_global_ids(*box, N)
    mask = inputs.box_boundary_mask(*box, N)
    if extra:  # masked nodes without any local copy
        mask = np.concatenate([mask, np.ones(extra, dtype=np.uint8)])
        ng += extra
    free = (mask == 0).astype(np.float64)

    def A(u):
        Y = orc.axlocal(G, orc.scatter(u, gid), N)
        return orc.gather(Y, gid, ng) * free

    dg = orc.gather(orc.element_diagonals(G, N), gid, ng)
    inv = np.where(free > 0, 1.0 / np.where(free > 0, dg, 1.0), 0.0)
    rng = np.random.default_rng(9)
    return V, gid, ng, mask, A, inv, rng.uniform(-1, 1, ng) * free, rng.uniform(-1, 1, ng)


@pytest.mark.parametrize("prec,tol", [("f64dw", 1e-9), ("fp32", 2e-4)])
@pytest.mark.parametrize("box,N,iters,precond,extra", [
    ((3, 3, 2), 7, 1, 1, 0), ((3, 3, 2), 7, 2, 1, 0), ((3, 3, 2), 7, 16, 1, 0), ((3, 3, 2), 7, 19, 1, 0),
    ((3, 3, 2), 7, 5, 0, 0), ((1, 1, 1), 6, 4, 1, 0), ((5, 3, 1), 4, 7, 1, 0), ((3, 2, 2), 5, 8, 1, 0),
    ((2, 2, 2), 10, 6, 1, 0), ((2, 1, 1), 15, 5, 1, 0), ((5, 5, 5), 2, 18, 1, 0), ((3, 3, 2), 7, 6, 1, 3)])
@pytest.mark.parametrize("kind", ["trilinear", "stored"])
def test_iterates(ax, orc, kind, box, N, iters, precond, extra, prec, tol):
    V, gid, ng, mask, A, inv, b, x0 = _problem(orc, box, N, extra)
    op = ax.Ax(torch.from_numpy(V).to(DEV), N, kind, prec)
    op.gs_setup(torch.from_numpy(gid).to(DEV), ng, torch.from_numpy(mask).to(DEV))
    bd = torch.from_numpy(b).to(DEV, op.dtype)
    for start in (np.zeros(ng), x0):
        ref = _cg(A, b, inv if precond else (mask == 0).astype(np.float64), np.where(mask == 1, 0.0, start), iters)
        x = torch.from_numpy(start).to(DEV, op.dtype)
        it, _, st = op.pcg_solve(bd, x, rtol=0.0, maxit=iters, precond=precond)
        assert st == ax.AX_ENOTCONV and it == iters
        err = np.max(np.abs(x.double().cpu().numpy() - ref)) / np.max(np.abs(ref))
        assert err <= tol, err


def test_stops_inside_a_block(ax, orc):
    # convergence in the middle of a captured block: the rest of the block is
    # idle and the last update of x is not lost
    V, gid, ng, mask, A, inv, b, _ = _problem(orc, (3, 3, 2), 5)
    op = ax.Ax(torch.from_numpy(V).to(DEV), 5, "trilinear", "f64dw")
    op.gs_setup(torch.from_numpy(gid).to(DEV), ng, torch.from_numpy(mask).to(DEV))
    bd = torch.from_numpy(b).to(DEV)
    for rtol in (1e-2, 1e-4, 1e-6, 1e-9):
        x = torch.zeros(ng, dtype=torch.float64, device=DEV)
        it, rr, st = op.pcg_solve(bd, x, rtol=rtol, maxit=500)
        assert st == ax.AX_OK and rr <= rtol
        true = np.linalg.norm(b - A(x.cpu().numpy())) / np.linalg.norm(b)
        assert abs(true - rr) <= 1e-10


@pytest.mark.parametrize("scale", [2.0 ** -200, 2.0 ** 150])
@pytest.mark.parametrize("N", [7, 11])
def test_far_from_unit_scale(ax, orc, N, scale):
    # a direction outside float32's exponent range: every block is read again,
    # scaled; CG is linear in b and powers of two are exact, so the iterates
    # scale with it
    V, gid, ng, mask, A, inv, b, _ = _problem(orc, (3, 2, 2), N)
    ref = _cg(A, b, inv, np.zeros(ng), 9)
    op = ax.Ax(torch.from_numpy(V).to(DEV), N, "trilinear", "f64dw")
    op.gs_setup(torch.from_numpy(gid).to(DEV), ng, torch.from_numpy(mask).to(DEV))
    x = torch.zeros(ng, dtype=torch.float64, device=DEV)
    op.pcg_solve(torch.from_numpy(b * scale).to(DEV), x, rtol=0.0, maxit=9)
    assert np.max(np.abs(x.cpu().numpy() / scale - ref)) <= 1e-9 * np.max(np.abs(ref))
