"""Operators on both sides of the lines where small meshes change from one thread
per node to line sweeps: a column alone (or four floats) against the same column
among others, which take the line sweeps on any mesh.

Bars: 1e-13 in FP64 and 2e-6 in float32 per column, both evaluations being off by a
few units of 1.1e-16 and 6e-8 of their largest terms.
"""
import pytest

pytestmark = pytest.mark.gpu

# degree, cells per axis (levels 1 and two nuclei add about 690 cells)
MESHES = [(2, 6), (2, 8), (2, 11), (3, 6), (3, 9), (3, 14), (3, 16), (4, 4), (4, 7), (4, 13), (4, 15)]


@pytest.fixture(scope="module", params=MESHES)
def mesh(request):
    import paper_2301_02387_gb300 as pkg
    p, nc = request.param
    return pkg.Mesh(-10.0, 10.0, nc, p, [((0.0, 0.0, 0.7), 1.0, 1), ((0.0, 0.0, -0.7), 1.0, 1)], 2.0)


def _worst(y, ref):
    return float(((y - ref).abs().pow(2).sum(0).sqrt() / ref.abs().pow(2).sum(0).sqrt()).max())


@pytest.mark.parametrize("k", [1, 2, 4, 8, 16])
def test_stiffness(mesh, k):
    import torch
    import paper_2301_02387_gb300 as pkg
    X = torch.randn((mesh.N, 36), generator=torch.Generator().manual_seed(k), dtype=torch.float64).cuda()
    ref = pkg.op_apply(mesh, pkg.OP_STIFF, X, torch.empty_like(X))[:, :k]
    x = X[:, :k].contiguous()
    assert _worst(pkg.op_apply(mesh, pkg.OP_STIFF, x, torch.empty_like(x)), ref) < 1e-13
    x = x.float()
    assert _worst(pkg.op_apply(mesh, pkg.OP_STIFF_F32, x, torch.empty_like(x)).double(), ref) < 2e-6


@pytest.mark.parametrize("n", [1, 2, 4, 8])
def test_h1(mesh, n):
    import torch
    import paper_2301_02387_gb300 as pkg
    E = (0.05, -0.02, 0.1)
    X = torch.randn((mesh.N, 9), generator=torch.Generator().manual_seed(n), dtype=torch.complex128).cuda()
    ref = pkg.op_apply(mesh, pkg.OP_H1, X, torch.empty_like(X), E=E)[:, :n]
    x = X[:, :n].contiguous()
    assert _worst(pkg.op_apply(mesh, pkg.OP_H1, x, torch.empty_like(x), E=E), ref) < 1e-13
    x = x.to(torch.complex64)
    assert _worst(pkg.op_apply(mesh, pkg.OP_H1_C64, x, torch.empty_like(x), E=E).to(torch.complex128), ref) < 2e-6
