"""Cell products from 1D tensor-product matrices (csrc/tensor_cells.cu) against the oracle's assembled
matrix: one cell, last blocks that are partly filled, every degree, hanging nodes in some and in all
blocks, and the vectors' constrained rows.

Tolerance as for the operator tests: 1e-12 relative in FP64 and 2e-5 in FP32 (round-off of about 10^3
terms per entry)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import assemble, mesh  # noqa: E402
from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

KINDS = {"stokes": 0, "stokes_a": 1, "pmass": 3}
CORNER, ALL = ((0.3, 0.3, 0.3), 0.3, 1), ((0.5, 0.5, 0.5), 0.45, 1)
CASES = [("stokes_a", 1, 1, None), ("stokes_a", 4, 1, None), ("stokes_a", 3, 2, None), ("stokes_a", 2, 3, None),
         ("stokes_a", 1, 4, None), ("stokes_a", 3, 1, CORNER), ("stokes_a", 2, 3, CORNER), ("stokes_a", 2, 4, CORNER),
         ("pmass", 5, 1, None), ("pmass", 2, 3, None), ("pmass", 2, 2, CORNER), ("pmass", 2, 3, CORNER),
         ("stokes", 1, 2, None), ("stokes", 3, 2, None), ("stokes", 3, 2, ALL), ("stokes", 1, 3, None),
         ("stokes", 3, 3, None), ("stokes", 2, 3, CORNER), ("stokes", 1, 4, None), ("stokes", 2, 4, CORNER)]


@pytest.mark.parametrize("kind,n,k,refine", CASES)
def test_product_equals_assembled_matrix(kind, n, k, refine):
    from paper_2603_29621_gb300 import api
    ctx = api.Context(0)
    m, f = api.Mesh(ctx, 3, n), mesh.uniform(3, n)
    if refine:
        m.refine_ball(*refine)
        f = mesh.refine_ball(f, *refine)
    p = api.Problem(ctx, m, kind=KINDS[kind], degree=k, nu=0.7, lambda_max=1.0)
    o = assemble.Problem(f, kind, k, nu=0.7)
    (xg, fg), (xo, fo) = p.support_points(), o.dofs.support_points()
    perm = inputs.match_dofs(xg, fg, xo, fo + 3 if kind == "pmass" else fo)
    x = inputs.uniform_vector(len(fo), seed=n)
    exp = o.vmult(x)
    xd = np.empty_like(x)
    xd[perm] = x
    for dt, tol in ((torch.float64, 1e-12), (torch.float32, 2e-5)):
        src = torch.tensor(xd, device="cuda", dtype=dt)
        got = p.vmult(src, torch.full_like(src, 7.0)).double().cpu().numpy()[perm]
        assert np.linalg.norm(got - exp) <= tol * np.linalg.norm(exp)
