"""Transfers between uniform levels (one tiled tensor-product launch, csrc/transfer_sep.cu) against the
tensor product of the dense 1D interpolation matrix: one tile, several tiles in y, tiles split in x
where the sums of a whole row do not fit, even (nested), odd (non-nested) and degree steps, one to four
components, 2D and 3D.

Tolerance: an entry is three nested sums of at most 11 products with weights of absolute row sum below
3, so its rounding error stays below 33 x 27 units in the last place of the largest input: 1e-13
relative to the largest output in FP64, 6e-5 in FP32."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

# (kind, dim, n, k, level): the step from `level` to the next coarser one
CASES = [("ns", 3, 2, 2, 0), ("ns", 3, 9, 2, 0), ("ns", 3, 22, 3, 0), ("ns", 3, 33, 2, 0), ("ns", 3, 36, 3, 0),
         ("ns", 3, 4, 3, 1), ("ns", 2, 45, 2, 0), ("ns", 2, 200, 3, 0), ("a", 3, 6, 4, 0), ("a", 3, 21, 1, 0),
         ("a", 2, 17, 3, 1)]


def _gll(k):
    return {1: [0, 1], 2: [0, .5, 1], 3: [0, .5 - .5 / math.sqrt(5), .5 + .5 / math.sqrt(5), 1],
            4: [0, .5 - .5 * math.sqrt(3 / 7), .5, .5 + .5 * math.sqrt(3 / 7), 1]}[k]


def _matrix(nf, kf, nc, kc):
    pos = [(i // kf + _gll(kf)[i % kf]) / nf for i in range(kf * nf + 1)]
    m, x = np.zeros((len(pos), kc * nc + 1)), _gll(kc)
    for i, p in enumerate(pos):
        c = min(int(math.floor(p * nc + 1e-12)), nc - 1)
        for a in range(kc + 1):
            m[i, kc * c + a] = np.prod([(p * nc - c - x[b]) / (x[a] - x[b]) for b in range(kc + 1) if b != a])
    return torch.tensor(m, device="cuda")


def _apply(m, u, dim):
    for d in range(dim):
        u = torch.movedim(torch.tensordot(m, u, dims=([1], [d])), 0, d)
    return u


@pytest.mark.parametrize("kind,dim,n,k,level", CASES)
def test_transfers_are_tensor_products(kind, dim, n, k, level):
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0)
    p = api.Problem(ctx, api.Mesh(ctx, dim, n), kind=L.STAB_NS if kind == "ns" else L.STOKES_A, degree=k, nu=1.0,
                    dt=1e-2 if kind == "ns" else 0.0, lambda_max=2.0)
    nf, nc = (round(p.info.level_cells[level + i] ** (1 / dim)) for i in (0, 1))
    kf, kc = p.info.level_degree[level], p.info.level_degree[level + 1]
    m, comp = _matrix(nf, kf, nc, kc), dim + 1 if kind == "ns" else dim

    def grid(v, nodes):
        return v.reshape([nodes] * dim + [comp]).clone()

    def inner(u):  # velocity of boundary nodes zeroed
        keep = torch.ones_like(u)
        for d in range(dim):
            e = keep.movedim(d, 0)
            e[0][..., :dim] = e[-1][..., :dim] = 0
        return u * keep
    for dt, tol in ((torch.float64, 1e-13), (torch.float32, 6e-5)):
        c = torch.tensor(inputs.uniform_vector(p.info.level_dofs[level + 1], seed=1), device="cuda", dtype=dt)
        f = torch.tensor(inputs.uniform_vector(p.info.level_dofs[level], seed=2), device="cuda", dtype=dt)
        exp = grid(f.double(), m.shape[0]) + inner(_apply(m, inner(grid(c.double(), m.shape[1])), dim))
        got = grid(p.prolongate_add(level, c, f.clone()).double(), m.shape[0])
        assert float((got - exp).abs().max()) <= tol * float(exp.abs().max())
        exp = inner(_apply(m.T, inner(grid(f.double(), m.shape[0])), dim))
        got = grid(p.restrict(level, f, torch.full_like(c, 9.0)).double(), m.shape[1])
        assert float((got - exp).abs().max()) <= tol * float(exp.abs().max())
