"""The FP64 stiffness of the cell pass against long double (points, weights and
derivatives of the basis included), on meshes without hanging points.

Bar: an entry is the sum of the parts of up to eight cells, each with three
roundings to float64 (its sum, its weight, their product), and seven additions;
together they stay below two units of 2^-53 of the norm.
"""
import numpy as np
import pytest

from oracle import mesh as omesh
from tests._match import coord_permutation

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _tables(p):
    """Gauss-Lobatto points and weights on [0, 1], stiffness matrix, in long double (Newton on P_p')."""
    def legendre(n, x):
        a, b = np.ones_like(x), x
        for k in range(2, n + 1):
            a, b = b, ((2 * k - 1) * x * b - (k - 1) * a) / LD(k)
        return b if n else a
    inner = np.sort(np.polynomial.legendre.Legendre.basis(p).deriv().roots().real) if p > 1 else []
    x = np.concatenate([[-1.0], inner, [1.0]]).astype(LD)
    for _ in range(6):
        q = x[1:-1]
        d = p * (legendre(p - 1, q) - q * legendre(p, q)) / (1 - q * q)
        x[1:-1] = q - d * (1 - q * q) / (2 * q * d - p * (p + 1) * legendre(p, q))
    w, xi, n = 1 / (LD(p * (p + 1)) * legendre(p, x) ** 2), (x + 1) / 2, p + 1
    D = np.zeros((n, n), LD)
    for j in range(n):
        for i in range(n):
            if i != j:
                D[i, j] = 1 / (xi[j] - xi[i])
                for k in range(n):
                    if k not in (i, j):
                        D[i, j] *= (xi[i] - xi[k]) / (xi[j] - xi[k])
    for i in range(n):
        D[i, i] = -sum(D[i, j] for j in range(n) if j != i)
    return w, D.T @ (w[:, None] * D)


@pytest.mark.parametrize("p,nc", [(1, 9), (2, 7), (3, 5), (4, 4)])
def test_stiffness_against_long_double(p, nc):
    import torch
    import paper_2301_02387_gb300 as pkg
    if np.finfo(LD).nmant < 63:
        pytest.skip("long double is float64 here")
    case = (-8.0, 8.0, nc, p, [((0.1, 0.2, 0.3), 1.0, 0)], 2.0)
    gm, om = pkg.Mesh(*case), omesh.Mesh(*case)
    perm = coord_permutation(gm.tables()[0], om.Xm)
    w, K = _tables(p)
    master = np.asarray(om.C.argmax(1)).ravel()
    x = np.random.default_rng(p).standard_normal((om.N, 4))
    n = p + 1
    u = x.astype(LD)[master][om.cell_pts].reshape(-1, n, n, n, 4)   # [cell][z][y][x]
    t = np.einsum("ij,nabjk->nabik", K, u) * w[:, None, None, None] * w[None, :, None, None]
    t += np.einsum("ij,najbk->naibk", K, u) * w[:, None, None, None] * w[None, None, :, None]
    t += np.einsum("ij,njabk->niabk", K, u) * w[None, :, None, None] * w[None, None, :, None]
    y = np.zeros((om.N, 4), LD)
    np.add.at(y, master[om.cell_pts].ravel(), (LD(16) / nc * t).reshape(-1, 4))
    X = torch.from_numpy(np.ascontiguousarray(x[perm])).cuda()
    Y = torch.empty_like(X)
    pkg.op_apply(gm, pkg.OP_STIFF, X, Y)
    err = Y.cpu().numpy().astype(LD) - y[perm]
    assert np.sqrt((err ** 2).sum()) <= 2.0 ** -52 * np.sqrt((y ** 2).sum())
