"""Block shapes that the small sizes of the operator tests do not reach, against the general kernel: full FP64
blocks of the line kernel, the larger FP64 blocks of the tensor-product cells with and without hanging
nodes, and cubic elements on the FP32 plane kernel in a launch of several problems.

Tolerances: those of the operator tests, 1e-12 in FP64 and 2e-5 in FP32 (round-off of about 10^3 terms per
entry); one problem and several in a launch are equal bit for bit."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def _compare(p, q):
    for dt, tol in ((torch.float64, 1e-12), (torch.float32, 2e-5)):
        x = torch.tensor(inputs.uniform_vector(p.info.n_dofs, seed=7), device="cuda", dtype=dt)
        got, want = p.vmult(x, torch.full_like(x, 7.0)), q.vmult(x, torch.empty_like(x))
        assert float((got - want).double().norm()) <= tol * float(want.double().norm())


# from 1,216 blocks of 128 / (k + 1)^2 cells on
@pytest.mark.parametrize("k,n", [(1, 35), (2, 27), (3, 23)])
def test_full_fp64_line_blocks(k, n):
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0)
    m = api.Mesh(ctx, 3, n)
    _compare(*(api.Problem(ctx, m, kind=L.STAB_NS, degree=k, nu=3e-2, dt=2e-2, lambda_max=2.0, recompute_frozen=r)
               for r in (0, 1)))


# FP64: blocks of 256 threads from 6,384 (degree 1) or 2,736 (degree 2) cells on; a budget that does not hold the
# products' buffer selects the general kernel
@pytest.mark.parametrize("kind,k,n,ball", [("a", 1, 19, 0), ("stokes", 2, 15, 0), ("a", 2, 13, 1), ("stokes", 2, 13, 1)])
def test_large_fp64_tensor_blocks(kind, k, n, ball):
    from paper_2603_29621_gb300 import _lib as L, api

    def build(limit):
        ctx = api.Context(0, hbm_budget_bytes=limit)
        m = api.Mesh(ctx, 3, n)
        if ball:
            m.refine_ball((0.5,) * 3, 0.25, ball)
        return ctx, api.Problem(ctx, m, kind=L.STOKES if kind == "stokes" else L.STOKES_A, degree=k, nu=0.7,
                                lambda_max=2.0)
    ctx, p = build(0)
    _compare(p, build(ctx.memory()[1] - 1)[1])


def test_cubic_plane_kernel_of_several_problems():
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0)
    ps = [api.Problem(ctx, api.Mesh(ctx, 3, n), kind=L.STAB_NS, degree=3, nu=1e-2, dt=1e-2, lambda_max=3.0,
                      mg_precision=L.FP32) for n in (17, 18, 17)]
    bs = [torch.tensor(inputs.uniform_vector(p.info.cycle_dofs, seed=i), device="cuda", dtype=torch.float32)
          for i, p in enumerate(ps)]
    xs = [torch.zeros_like(b) for b in bs]
    api.batch_vcycle(ps, bs, xs)
    for p, b, x in zip(ps, bs, xs):
        assert torch.equal(x, p.vcycle(b, torch.zeros_like(b)))
