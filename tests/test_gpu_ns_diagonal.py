"""Diagonal of the stabilised operator on uniform 3D levels (summed from the stored point values), and of the
colour-ordered one in 2D, against the products of unit vectors."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,k,terms,div_sign", [
    (3, 1, 1, 0, 0.0), (3, 1, 3, 0, 0.0), (3, 2, 2, 0, 0.0), (3, 3, 1, 0, 0.0), (3, 3, 3, 0, 0.0), (3, 4, 2, 0, 0.0),
    (3, 13, 2, 0, 0.0),                    # several blocks of point values a cell row
    (3, 3, 2, 0x3F, 0.0), (3, 3, 2, 0x61, 1.0), (3, 3, 3, 0x29, -1.0),   # without the viscous, convection, SUPG terms
    (2, 5, 2, 0, 0.0), (2, 40, 3, 0, 0.0), (2, 96, 2, 0, 0.0),           # one launch over all cells against colours
])
def test_diagonal_is_that_of_the_products(dim, n, k, terms, div_sign):
    """Both evaluate the same integrals in a different order; an entry is a sum of up to 8 (k + 1)^3 points with
    terms of both signs, none larger than the diagonal of the whole by more than a few times, so 64 units in
    the last place of the largest entry bound the difference (1e-13 covers FP64)."""
    from paper_2603_29621_gb300 import _lib as L
    from paper_2603_29621_gb300 import api

    ctx = api.Context(0)
    p = api.Problem(ctx, api.Mesh(ctx, dim, n), kind=L.STAB_NS, degree=k, nu=1e-2, dt=1e-2, terms=terms,
                    div_sign=div_sign, lambda_max=3.0)
    rng = np.random.default_rng(5)
    m = p.info.n_dofs
    pick = np.unique(np.concatenate([np.arange(min(m, dim + 1)), rng.integers(0, m, 60), [m - 1]]))
    for dtype, eps in ((torch.float64, 1e-13), (torch.float32, 64 * 2.0 ** -24)):
        diag = torch.empty(m, dtype=dtype, device="cuda")
        p.diagonal(diag)
        e, y = torch.zeros(m, dtype=dtype, device="cuda"), torch.empty(m, dtype=dtype, device="cuda")
        want = torch.empty(len(pick), dtype=dtype, device="cuda")
        for j, i in enumerate(pick):
            e[i] = 1
            want[j] = p.vmult(e, y)[i]
            e[i] = 0
        got = diag[torch.as_tensor(pick, device="cuda")]
        free = torch.as_tensor(~np.isin(pick, p.constrained(L.OP_SYSTEM)), device="cuda")
        # velocity and pressure entries differ in size: each compared with the largest of its own kind
        comp = torch.as_tensor(pick % (dim + 1) == dim, device="cuda")
        for kind in (comp, ~comp):
            scale = float(want[kind & free].abs().max()) if bool((kind & free).any()) else 1.0
            assert float((got - want)[kind].abs().max()) <= eps * max(scale, 1.0 if bool((kind & ~free).any()) else 0.0)
