"""ax_diag (element diagonals from the vertices) against the CPU oracle's
diagonals from its own factors, at every shape of the kernel: several elements
per CTA with a ragged last CTA, exactly one element, one element per CTA.

Tolerance: a diagonal entry is a sum of about 3 N1 + 3 products of positive
size, each factor good to a few roundings of a well-conditioned element
(perturbation 0.1 h), so its FP64 error is below (3 N1 + 30) 2^-53 of the
largest entry, under 1e-14 for N1 <= 16; 1e-13 leaves the margin of the
existing test.  float32 results add one rounding, 2^-24."""
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


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N,box", [(1, (33, 1, 1)), (1, (1, 1, 1)), (2, (5, 3, 1)), (3, (3, 3, 1)), (4, (3, 2, 1)),
                                   (5, (2, 2, 1)), (6, (3, 1, 1)), (7, (3, 1, 1)), (9, (2, 1, 1)), (10, (2, 2, 1)),
                                   (11, (2, 1, 1)), (12, (1, 1, 1)), (14, (2, 1, 1)), (15, (2, 1, 1))])
def test_diagonal_every_shape(ax, orc, N, box, prec):
    V = inputs.box_vertices(*box, perturb=0.1, seed=3)
    # the boundary of a thin box is not perturbed: skew it so that no factor vanishes
    V = V @ np.array([[1.0, 0.2, 0.1], [0.0, 1.1, 0.3], [0.0, 0.0, 0.9]]).T
    G, bad = orc.factors(V, N)
    assert bad == 0
    ref = orc.element_diagonals(G, N)
    op = ax.Ax(torch.from_numpy(np.ascontiguousarray(V)).to(DEV), N, "trilinear", prec)
    d = op.ax_diag(torch.full(ref.shape, float("nan"), dtype=op.dtype, device=DEV)).double().cpu().numpy()
    tol = 1e-13 if prec == "fp64" else 2.0 ** -24
    assert np.max(np.abs(d - ref)) <= tol * np.abs(ref).max()
