"""Handles of a context destroyed in any order (a garbage collector destroys a cycle's members in any)."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [(0, 1, 2, 3), (3, 2, 1, 0), (0, 3, 1, 2), (2, 0, 1, 3)])
def test_context_lives_as_long_as_what_was_made_with_it(order):
    from paper_2603_29621_gb300 import _lib as L, api

    ctx = api.Context(0)
    m = api.Mesh(ctx, 2, 4)
    p = api.Problem(ctx, m, kind=L.STOKES, degree=2, nu=1.0)
    st = api.SpaceTime(p, 1, 0.1)
    handles = [ctx, m, p, st]
    for i in order:
        if i == 2 and st.h:  # a slab refers to its problem
            st.close()
        handles[i].close()
        if p.h:
            x = torch.ones(p.info.n_dofs, dtype=torch.float64, device="cuda")
            p.vmult(x, torch.empty_like(x))
    assert float(torch.ones(3, device="cuda").sum()) == 3.0  # no error left behind
