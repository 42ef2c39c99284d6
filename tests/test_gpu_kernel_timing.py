"""Kernel timing covers every launch of a product: the cell launch and the node pass where the level has
them, the colour launches elsewhere."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,dim,n,ball,opts,launches", [
    ("ns", 3, 9, 0, {}, 2), ("ns", 3, 3, 1, {}, 2), ("stokes", 3, 4, 0, {}, 2), ("stokes", 2, 8, 0, {}, 2),
    ("ns", 3, 17, 0, dict(recompute_frozen=1), 8)])
def test_every_launch_of_a_product_is_timed(kind, dim, n, ball, opts, launches):
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0)
    m = api.Mesh(ctx, dim, n)
    if ball:
        m.refine_ball((0.5,) * 3, 0.3, ball)
    p = api.Problem(ctx, m, kind=L.STAB_NS if kind == "ns" else L.STOKES, degree=2, nu=1.0,
                    dt=1e-2 if kind == "ns" else 0.0, lambda_max=2.0, **opts)
    for dt in (torch.float32, torch.float64):
        x = torch.ones(p.info.n_dofs, device="cuda", dtype=dt)
        y = torch.empty_like(x)
        p.vmult(x, y)
        p.kernel_timing(1)
        for _ in range(3):
            p.vmult(x, y)
        ms, count = p.kernel_timing(2)
        p.kernel_timing(0)
        assert count == 3 * launches and ms > 0
