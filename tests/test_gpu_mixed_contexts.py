"""One high-precision context whose mixed solves use several low-precision
contexts, each destroyed before the next is made: their arrays have the same
sizes, so the allocator may hand the next one the addresses of the last, and the
iterations that the high-precision context keeps captured must not be replayed
for another operator.  Every solve must be the one of a fresh pair of contexts:
the same iteration counts and, the sums being in a fixed order, the same bits."""
import numpy as np
import pytest

from paper_2504_07042_gb300 import inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N, n = 5, 4


@pytest.fixture(scope="module")
def ax():
    from paper_2504_07042_gb300 import build

    build.build()
    from paper_2504_07042_gb300 import ax as _ax

    return _ax


@pytest.mark.parametrize("kind", ["trilinear", "partial"])
def test_each_solve_uses_its_own_context(ax, kind):
    V = torch.from_numpy(inputs.box_vertices(n, n, n, perturb=0.1, seed=3)).to(DEV)
    gid, ng = inputs.box_global_ids(n, n, n, N)
    gid, mask = torch.from_numpy(gid).to(DEV), torch.from_numpy(inputs.box_boundary_mask(n, n, n, N)).to(DEV)
    b = torch.from_numpy(np.random.default_rng(4).uniform(-1, 1, ng)).to(DEV)

    def high():
        hi = ax.Ax(V, N, kind, "f64dw")
        hi.gs_setup(gid, ng, mask)
        return hi

    def solve(hi, prec):
        lo = ax.Ax(V, N, kind, prec)
        x = torch.zeros_like(b)
        outer, inner, _, st = hi.pcg_solve_mixed(lo, b, x, rtol=1e-10, inner_rtol=1e-2, max_outer=100)
        assert st == ax.AX_OK
        lo.ax_destroy()
        return outer, inner, x

    kept, precs = high(), ("fp32", "bf16", "tf32", "fp16", "tf32", "fp32")
    got = [solve(kept, prec) for prec in precs]
    for prec, (outer, inner, x) in zip(precs, got):
        outer_ref, inner_ref, x_ref = solve(high(), prec)
        assert (outer, inner) == (outer_ref, inner_ref) and torch.equal(x, x_ref), prec
