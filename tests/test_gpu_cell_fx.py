"""The FP64 cell pass on the integer pipe at its edges: column counts around the
16 of a block and its tails, columns of very different size, tiny and huge
values, zeros and non-finite entries, on meshes whose last block holds fewer
cells.  Reference: the oracle's assembled matrices; bar 1e-10 per column, the
FP64 parity bar of the operators (two passes sum in different orders)."""
import numpy as np
import pytest

from oracle import fem, mesh as omesh
from tests._match import assert_close, coord_permutation

pytestmark = pytest.mark.gpu

MESHES = [
    (-6.0, 6.0, 3, 1, [((0.3, 0.1, 0.2), 1.0, 2)], 2.0),
    (-6.0, 6.0, 3, 2, [((0.3, 0.1, 0.2), 1.0, 1)], 2.0),
    (-5.0, 5.0, 2, 3, [((0.0, 0.0, 0.0), 2.0, 1)], 2.0),
    (-5.0, 5.0, 2, 4, [((0.0, 0.0, 0.0), 2.0, 1)], 1.0),
]


@pytest.fixture(scope="module", params=range(len(MESHES)))
def space(request):
    import paper_2301_02387_gb300 as pkg
    gm, om = pkg.Mesh(*MESHES[request.param]), omesh.Mesh(*MESHES[request.param])
    return gm, om, fem.Operators(om), coord_permutation(gm.tables()[0], om.Xm)


def _apply(gm, kind, xo, perm, E=None):
    import torch
    import paper_2301_02387_gb300 as pkg
    x = torch.from_numpy(np.ascontiguousarray(xo[perm])).cuda()
    y = torch.empty_like(x)
    pkg.op_apply(gm, kind, x, y, E=E)
    return y.cpu().numpy()


@pytest.mark.parametrize("k", [1, 3, 9, 16, 17, 25, 36, 64])
@pytest.mark.parametrize("spread", [0.0, 30.0])
def test_stiffness_columns(space, k, spread):
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    rng = np.random.default_rng(k)
    x = rng.standard_normal((om.N, k)) * 10.0 ** (spread * (np.arange(k) / k - 0.5))
    got = _apply(gm, pkg.OP_STIFF, x, perm)
    assert_close(got, op.stiffness_apply(x)[perm], 1e-10, axis=0, what="stiffness")


@pytest.mark.parametrize("n", [1, 4, 8, 9, 20])
def test_h1_columns(space, n):
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    rng = np.random.default_rng(n)
    x = rng.standard_normal((om.N, n)) + 1j * rng.standard_normal((om.N, n))
    x[:, 0] *= 1e-12
    E = (0.05, -0.02, 0.1)
    assert_close(_apply(gm, pkg.OP_H1, x, perm, E), op.h1_apply(x, E=E)[perm], 1e-10, axis=0, what="H1")


@pytest.mark.parametrize("power", [-900, 900])
def test_power_of_two_scaling(space, power):
    """A scaling by a power of two is exact up to the order of the atomic sums (1e-12)."""
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    x = np.random.default_rng(0).standard_normal((om.N, 5))
    a, b = _apply(gm, pkg.OP_STIFF, x, perm), _apply(gm, pkg.OP_STIFF, x * 2.0 ** power, perm)
    assert_close(b * 2.0 ** -power, a, 1e-12, axis=0, what="scaled stiffness")


def test_zeros_and_non_finite(space):
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    x = np.random.default_rng(1).standard_normal((om.N, 3))
    x[:, 1] = 0.0
    got = _apply(gm, pkg.OP_STIFF, x, perm)
    assert np.all(got[:, 1] == 0.0)
    x[om.N // 2, 2] = np.nan
    got = _apply(gm, pkg.OP_STIFF, x, perm)
    assert np.isnan(got[:, 2]).any() and np.isfinite(got[:, :2]).all()
