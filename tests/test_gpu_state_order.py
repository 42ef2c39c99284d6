"""A product enqueued directly behind a new linearisation state reads that state's point values: levels of
every product path, 2D levels that defer in FP32 only (between 2^19 and 2^20 contributions) among them."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,k,ball,recompute", [(2, 300, 2, 0, 0), (2, 16, 2, 0, 0), (2, 400, 2, 0, 0),
                                                    (3, 5, 2, 0, 0), (3, 20, 2, 0, 0), (3, 4, 2, 1, 0),
                                                    (3, 5, 2, 0, 1)])
def test_product_behind_a_new_state(dim, n, k, ball, recompute):
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0)
    m = api.Mesh(ctx, dim, n)
    if ball:
        m.refine_ball((0.5,) * 3, 0.3, ball)
    p = api.Problem(ctx, m, kind=L.STAB_NS, degree=k, nu=1e-2, dt=1e-2, lambda_max=2.0, recompute_frozen=recompute,
                    mg_precision=L.FP32)
    size = p.info.n_dofs
    states = [torch.tensor(inputs.uniform_vector(size, seed=s), device="cuda") for s in (1, 2)]
    for dt in (torch.float32, torch.float64):
        x = torch.tensor(inputs.uniform_vector(size, seed=3), device="cuda", dtype=dt)
        for u in states:
            got, want = torch.empty_like(x), torch.empty_like(x)
            p.set_state(1e-2, 1.5, u)
            p.vmult(x, got)
            torch.cuda.synchronize()
            p.vmult(x, want)
            assert torch.equal(got, want)
