"""The HBM budget decides how products are laid out, not whether a problem exists: one that fits without the
buffer between a product's launches and its tables is created without them and gives the same results
(products and transfers on every level, to the bounds of the operator tests); a budget below that is
refused, and nothing stays allocated."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

# kind, dim, n, degree, refinements
CASES = [("ns", 3, 9, 2, 0), ("ns", 3, 17, 1, 0), ("ns", 3, 5, 3, 0), ("ns", 3, 4, 2, 1), ("ns", 2, 24, 2, 0),
         ("a", 3, 9, 1, 0), ("a", 3, 5, 2, 1), ("stokes", 3, 5, 2, 1), ("stokes", 3, 6, 3, 0), ("stokes", 2, 16, 2, 0)]


def _problem(limit, kind, dim, n, k, ball):
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0, hbm_budget_bytes=limit)
    m = api.Mesh(ctx, dim, n)
    if ball:
        m.refine_ball((0.5,) * 3, 0.3, ball)
    p = api.Problem(ctx, m, kind={"ns": L.STAB_NS, "a": L.STOKES_A, "stokes": L.STOKES}[kind], degree=k, nu=0.1,
                    dt=1e-2 if kind == "ns" else 0.0, lambda_max=2.0, mg_precision=L.FP32)
    return ctx, p


@pytest.mark.parametrize("kind,dim,n,k,ball", CASES)
def test_a_tight_budget_changes_the_layout_only(kind, dim, n, k, ball):
    from paper_2603_29621_gb300 import _lib as L
    ctx, p = _problem(0, kind, dim, n, k, ball)
    full = ctx.memory()[0]
    tight, q = _problem(full - 1, kind, dim, n, k, ball)
    assert tight.memory()[1] <= full - 1
    for dt, tol in ((torch.float64, 1e-12), (torch.float32, 2e-5)):
        x = torch.tensor(inputs.uniform_vector(p.info.n_dofs, seed=1), device="cuda", dtype=dt)
        want, got = p.vmult(x, torch.empty_like(x)), q.vmult(x, torch.empty_like(x))
        assert float((got - want).double().norm()) <= tol * float(want.double().norm())
        # every level's product, and the transfers between them
        for level in range(p.info.n_levels):
            x = torch.tensor(inputs.uniform_vector(p.info.level_dofs[level], seed=2), device="cuda", dtype=dt)
            want, got = (r.vmult(x, torch.empty_like(x), which=level) for r in (p, q))
            assert float((got - want).double().norm()) <= tol * float(want.double().norm())
            if level + 1 == p.info.n_levels:
                break
            c = torch.tensor(inputs.uniform_vector(p.info.level_dofs[level + 1], seed=3), device="cuda", dtype=dt)
            for want, got in ((r.restrict(level, x, torch.empty_like(c)) for r in (p, q)),
                              (r.prolongate_add(level, c, x.clone()) for r in (p, q))):
                assert float((got - want).double().norm()) <= tol * float(want.double().norm())
    with pytest.raises(L.MfnsError) as e:
        _problem(full // 2, kind, dim, n, k, ball)
    assert e.value.code == L.ERR_BUDGET


@pytest.mark.parametrize("kind,k,n", [("a", 2, 6), ("a", 3, 4), ("ns", 2, 7)])
def test_batches_of_both_layouts(kind, k, n):
    """A problem with the products' buffer and one without it in a batch: each gives what it gives alone, bit for
    bit (their products round differently, so they must not share launches)."""
    from paper_2603_29621_gb300 import _lib as L, api
    ctx, p = _problem(0, kind, 3, n, k, 0)
    tight = api.Context(0, hbm_budget_bytes=2 * ctx.memory()[0] - 1)
    ps = [api.Problem(tight, api.Mesh(tight, 3, n), kind=L.STAB_NS if kind == "ns" else L.STOKES_A, degree=k, nu=0.1,
                      dt=1e-2 if kind == "ns" else 0.0, lambda_max=2.0, mg_precision=L.FP32) for _ in range(2)]
    assert tight.memory()[0] < 2 * ctx.memory()[0]
    for dt in (torch.float64, torch.float32):
        bs = [torch.tensor(inputs.uniform_vector(p.info.cycle_dofs, seed=s), device="cuda", dtype=dt) for s in (4, 5)]
        xs = [torch.zeros_like(b) for b in bs]
        api.batch_vcycle(ps, bs, xs)
        for q, b, x in zip(ps, bs, xs):
            assert torch.equal(x, q.vcycle(b, torch.zeros_like(b)))


def test_a_refused_problem_leaves_nothing_allocated():
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0, hbm_budget_bytes=1 << 20)
    with pytest.raises(L.MfnsError):
        api.Problem(ctx, api.Mesh(ctx, 3, 8), kind=L.STOKES, degree=2, nu=1.0, lambda_max=1.0)
    assert ctx.memory()[0] == 0


def test_space_time_multigrid_in_a_tight_budget():
    from paper_2603_29621_gb300 import _lib as L, api

    def build(limit):
        ctx = api.Context(0, hbm_budget_bytes=limit)
        p = api.Problem(ctx, api.Mesh(ctx, 2, 8), kind=L.STOKES, degree=2, nu=1.0, lambda_max=2.0)
        st = api.SpaceTime(p, 1, 0.1)
        st.mg_build()
        return ctx, st
    ctx, st = build(0)
    tight, sq = build(ctx.memory()[1] - 1)
    assert tight.memory()[1] < ctx.memory()[1]
    x = torch.tensor(inputs.uniform_vector(st.Q * st.n, seed=3), device="cuda")
    want, got = st.vcycle(x, torch.zeros_like(x)), sq.vcycle(x, torch.zeros_like(x))
    assert float((got - want).norm()) <= 1e-10 * float(want.norm())
