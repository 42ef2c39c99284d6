"""Rounding of the FP64 cell products from 1D tensor-product matrices (csrc/tensor_cells.cu), against the
assembled operator in extended precision with exact 1D integrals.

Bound: 3e-16 of the result in the l2 norm, 2.7 units of rounding u = 1.1e-16.  An entry is a sum of products of
three table entries, each rounded to nearest (at most u, 0.6 u rms, so about u for the product), through
three contractions of up to 5 terms whose roundings add in quadrature (another 1.5 u), on meshes of a power
of two cells, where the scaling by h is exact."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_29621_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _nodes(k):
    five, tf = np.sqrt(LD(5)), np.sqrt(LD(3) / LD(7))
    return {1: [LD(-1), LD(1)], 2: [LD(-1), LD(0), LD(1)], 3: [LD(-1), -1 / five, 1 / five, LD(1)],
            4: [LD(-1), -tf, LD(0), tf, LD(1)]}[k]


def _basis(k):
    t, out = _nodes(k), []
    for a in range(k + 1):
        c = np.array([LD(1)])
        for m in range(k + 1):
            if m != a:
                c = (np.concatenate([[LD(0)], c]) - np.concatenate([t[m] * c, [LD(0)]])) / (t[a] - t[m])
        out.append(c)
    return out


def _matrices(k, n):
    """1D mass and stiffness of n cells of width 1/n."""
    b = _basis(k)
    d = [np.array([2 * i * c[i] for i in range(1, k + 1)], LD) for c in b]

    def integral(p, q):
        return sum((p[i] * q[j] / (i + j + 1) for i in range(len(p)) for j in range(len(q)) if (i + j) % 2 == 0), LD(0))
    M, K = np.zeros((k * n + 1,) * 2, LD), np.zeros((k * n + 1,) * 2, LD)
    for c in range(n):
        for i in range(k + 1):
            for j in range(k + 1):
                M[k * c + i, k * c + j] += integral(b[i], b[j]) / n
                K[k * c + i, k * c + j] += integral(d[i], d[j]) * n
    return M, K


def _apply(mats, u):
    for d, m in enumerate(mats):
        u = np.moveaxis(np.tensordot(m, np.moveaxis(u, d, 0), axes=(1, 0)), 0, d)
    return u


def test_reference_matrices_are_exact():
    m, k = _matrices(2, 1)
    for i, j, mass, stiff in ((0, 0, Fraction(2, 15), Fraction(7, 3)), (0, 1, Fraction(1, 15), Fraction(-8, 3)),
                              (1, 1, Fraction(8, 15), Fraction(16, 3)), (0, 2, Fraction(-1, 30), Fraction(1, 3))):
        assert abs(float(m[i, j]) - float(mass)) <= 1e-16 and abs(float(k[i, j]) - float(stiff)) <= 1e-15


@pytest.mark.parametrize("kind,k,n", [("a", 1, 8), ("a", 2, 4), ("a", 3, 4), ("a", 4, 4), ("pmass", 1, 8),
                                      ("pmass", 2, 4), ("pmass", 3, 4)])
def test_products_round_like_exact_tables(kind, k, n):
    from paper_2603_29621_gb300 import _lib as L, api
    ctx = api.Context(0)
    p = api.Problem(ctx, api.Mesh(ctx, 3, n), kind=L.STOKES_A if kind == "a" else L.PMASS, degree=k, nu=1.0,
                    lambda_max=1.0)
    comp, nodes = 3 if kind == "a" else 1, k * n + 1
    x = inputs.uniform_vector(p.info.n_dofs, seed=k)
    x[p.constrained(L.OP_SYSTEM)] = 0
    got = p.vmult(torch.tensor(x, device="cuda"), torch.empty(len(x), device="cuda", dtype=torch.float64))
    M, K = _matrices(k, n)
    u = x.astype(LD).reshape(nodes, nodes, nodes, comp)
    want = sum(_apply(m, u) for m in ([K, M, M], [M, K, M], [M, M, K])) if kind == "a" else _apply([M, M, M], u)
    want = want.reshape(-1).copy()
    want[p.constrained(L.OP_SYSTEM)] = 0
    e = got.cpu().numpy().astype(LD) - want
    assert float(np.sqrt((e * e).sum() / (want * want).sum())) <= 3e-16
