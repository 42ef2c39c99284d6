"""The stabilised operator on uniform 3D levels (cell rows and a node pass, csrc/ns_lines.cuh) against the
general cell kernel, which the option recompute_frozen selects: sizes around the blocks' edges (one
cell, a cell row broken by a block, a last block that is partly filled, full FP32 blocks on the plane
kernel), every degree, single terms and both signs of the continuity row.

Tolerances: both paths sum the same terms in another order.  An output entry adds at most 8 cells x 64
points x 40 products, so rounding stays below a few hundred units in the last place of the largest
summand: 1e-12 relative in FP64 and 2e-5 in FP32, the bounds of the operator tests."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (1, 2), (1, 7), (1, 17), (2, 1), (2, 3), (2, 5), (2, 11), (2, 17), (3, 1), (3, 2), (3, 5), (3, 17)]


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_29621_gb300 import api
    return api.Context(0)


def _pair(ctx, n, k, **kw):
    from paper_2603_29621_gb300 import _lib as L, api
    m = api.Mesh(ctx, 3, n)
    d = dict(kind=L.STAB_NS, degree=k, nu=3e-2, dt=2e-2, lambda_max=2.0, **kw)
    return [api.Problem(ctx, m, recompute_frozen=r, **d) for r in (0, 1)]


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("k,n", SIZES)
def test_product_equals_general_kernel(ctx, k, n):
    new, old = _pair(ctx, n, k)
    x = torch.tensor(inputs.uniform_vector(new.info.n_dofs, seed=n), device="cuda")
    y = old.vmult(x, torch.zeros_like(x))
    assert _rel(new.vmult(x, torch.full_like(x, 7.0)), y) <= 1e-12
    assert _rel(new.vmult(x.float(), torch.full_like(x, 7.0).float()), y) <= 2e-5


@pytest.mark.parametrize("terms,sign", [(32 + 1, 0.0), (32 + 2, -1.0), (32 + 4, 0.0), (32 + 8, 0.0), (32 + 16, 2.0),
                                        (32, -1.0), (32 + 64, 0.0), (127, -1.0), (127 - 2, 0.0), (127 - 8, 0.0)])
def test_terms_and_sign(ctx, terms, sign):  # PSPG always on: without it the coarse system is singular
    new, old = _pair(ctx, 5, 2, terms=terms, div_sign=sign)
    x = torch.tensor(inputs.uniform_vector(new.info.n_dofs, seed=3), device="cuda")
    y = old.vmult(x, torch.zeros_like(x))
    assert _rel(new.vmult(x, torch.zeros_like(x)), y) <= 1e-12
    assert _rel(new.vmult(x.float(), torch.zeros_like(x).float()), y) <= 2e-5


@pytest.mark.parametrize("prec,tol", [("f64", 1e-11), ("f32", 2e-5)])
@pytest.mark.parametrize("k,n", [(1, 9), (2, 6), (2, 17), (3, 4)])
@pytest.mark.parametrize("smoother", [1, 2])
def test_smoother_update_in_the_node_pass(ctx, prec, tol, k, n, smoother):
    new, old = _pair(ctx, n, k, smoother=smoother, smoother_degree=4)
    dt = torch.float64 if prec == "f64" else torch.float32
    b, x0 = (torch.tensor(inputs.uniform_vector(new.info.n_dofs, seed=s), device="cuda", dtype=dt) for s in (4, 5))
    for zero in (True, False):
        got, exp = x0.clone(), x0.clone()
        new.smooth(0, b, got, x_is_zero=zero)
        old.smooth(0, b, exp, x_is_zero=zero)
        assert _rel(got, exp) <= tol
