"""Vectors that do not start on a 16-byte boundary (views of a longer tensor) on the levels whose kernels
access four components at a time: the smoother and the transfers take them and give the result of
aligned vectors bit for bit; calls whose operand would be read by a product refuse them."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")

from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def _vec(n, seed, dt):
    return torch.tensor(inputs.uniform_vector(n, seed=seed), device="cuda", dtype=dt)


def _off(v):  # the same values, one entry behind a boundary
    return torch.cat([v.new_zeros(1), v])[1:]


@pytest.fixture(scope="module")
def problems():
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0)
    return [api.Problem(ctx, api.Mesh(ctx, 3, 5), kind=L.STAB_NS, degree=2, nu=1e-2, dt=1e-2, lambda_max=2.0,
                        smoother_degree=3, recompute_frozen=r) for r in (0, 1)]


@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("which", [0, 1])
def test_smoother_and_transfers_take_offset_views(problems, which, dt):
    p = problems[which]
    nf, nc = p.info.level_dofs[0], p.info.level_dofs[1]
    b, x, c = _vec(nf, 1, dt), _vec(nf, 2, dt), _vec(nc, 3, dt)
    for zero in (True, False):
        want = p.smooth(0, b, x.clone(), x_is_zero=zero)
        for bb, xx in ((_off(b), x.clone()), (b, _off(x)), (_off(b), _off(x))):
            assert torch.equal(p.smooth(0, bb, xx, x_is_zero=zero), want)
    want = p.restrict(0, b, torch.zeros_like(c))
    assert torch.equal(p.restrict(0, _off(b), _off(torch.ones_like(c))), want)
    want = p.prolongate_add(0, c, x.clone())
    assert torch.equal(p.prolongate_add(0, _off(c), _off(x)), want)


def test_operands_of_products_are_refused(problems):
    from paper_2603_29621_gb300 import _lib as L, api
    p = problems[0]
    n = p.info.level_dofs[0]
    b, x = _vec(n, 1, torch.float32), _off(_vec(n, 2, torch.float32))
    calls = [lambda: p.vmult(x, torch.zeros_like(b)), lambda: api.batch_vcycle([p], [b], [x]),
             lambda: L.check(p.lib.mfns_smooth_noalloc(p.h, 0, L.FP32, C.c_void_p(b.data_ptr()),
                                                       C.c_void_p(x.data_ptr()), n, 0, None))]
    for call in calls:
        with pytest.raises(L.MfnsError) as e:
            call()
        assert e.value.code == L.ERR_ARG
