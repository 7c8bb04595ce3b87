"""Entry by entry accuracy of the FP64 cell pass on the integer pipe: values whose
size differs from node to node within a cell, values near the bottom of the
float64 range, and infinities, which stay on the lines of their node.

Bar: with B = |C|^T (sum_K |A_K|) |C| |x| the float64 evaluation is off by at most
k 2^-53 B in each entry, k the number of roundings on the way to it (3 (p + 1)
products, the weights, the constraint rows in and out, up to eight cells: below
100); the kernel and the oracle may each use that: 200 * 2^-53 B.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import fem, mesh as omesh
from tests._match import assert_close, coord_permutation

pytestmark = pytest.mark.gpu

MESHES = [
    (-6.0, 6.0, 3, 1, [((0.3, 0.1, 0.2), 1.0, 2)], 2.0),
    (-6.0, 6.0, 3, 2, [((0.3, 0.1, 0.2), 1.0, 1)], 2.0),
    (-5.0, 5.0, 2, 3, [((0.0, 0.0, 0.0), 2.0, 1)], 2.0),
    (-5.0, 5.0, 2, 4, [((0.0, 0.0, 0.0), 2.0, 1)], 1.0),
]
BAR = 200.0 * 2.0 ** -53


@pytest.fixture(scope="module", params=range(len(MESHES)))
def space(request):
    import paper_2301_02387_gb300 as pkg
    gm, om = pkg.Mesh(*MESHES[request.param]), omesh.Mesh(*MESHES[request.param])
    op = fem.Operators(om)
    A_hat, _ = fem.cell_matrices(om.p)
    nn, ncell = (om.p + 1) ** 3, len(om.lev)
    vals = (om.h[:, None, None] * np.abs(A_hat)[None]).reshape(ncell, -1).ravel()
    A_abs = sp.csr_matrix((vals, (np.repeat(om.cell_pts, nn, axis=1).ravel(), np.tile(om.cell_pts, (1, nn)).ravel())),
                          shape=(om.nf, om.nf))
    A_abs = (abs(om.C).T @ A_abs @ abs(om.C)).tocsr()
    return gm, om, op, A_abs, coord_permutation(gm.tables()[0], om.Xm)


def _apply(gm, kind, xo, perm, E=None):
    import torch
    import paper_2301_02387_gb300 as pkg
    x = torch.from_numpy(np.ascontiguousarray(xo[perm])).cuda()
    y = torch.empty_like(x)
    pkg.op_apply(gm, kind, x, y, E=E)
    return y.cpu().numpy()


@pytest.mark.parametrize("spread", [6, 30, 200])
def test_stiffness_entry_by_entry(space, spread):
    import paper_2301_02387_gb300 as pkg
    gm, om, op, A_abs, perm = space
    rng = np.random.default_rng(spread)
    x = rng.standard_normal((om.N, 5)) * 2.0 ** (-spread * rng.random((om.N, 5)))
    err = np.abs(_apply(gm, pkg.OP_STIFF, x, perm) - op.stiffness_apply(x)[perm])
    assert np.all(err <= BAR * (A_abs @ np.abs(x))[perm])


@pytest.mark.parametrize("spread", [6, 30, 200])
def test_h1_entry_by_entry(space, spread):
    """Real and imaginary parts are columns of their own."""
    import paper_2301_02387_gb300 as pkg
    gm, om, op, A_abs, perm = space
    rng = np.random.default_rng(spread + 1)
    x = (rng.standard_normal((om.N, 3)) + 1j * rng.standard_normal((om.N, 3))) * 2.0 ** (-spread * rng.random((om.N, 3)))
    E = (0.05, -0.02, 0.1)
    got, ref = _apply(gm, pkg.OP_H1, x, perm, E), op.h1_apply(x, E=E)[perm]
    f = np.abs(op.V_f) + np.abs(om.X) @ np.abs(np.array(E))
    B = 0.5 * A_abs + abs(om.C).T @ sp.diags(op.m_f * f) @ abs(om.C)
    for part in (np.real, np.imag):
        b = (B @ np.abs(part(x) * op.interior[:, None])) * (op.interior / op.ML)[:, None]
        assert np.all(np.abs(part(got) - part(ref)) <= BAR * b[perm])


def test_values_near_the_bottom_of_the_range(space):
    """A scaling by 2^-1000 is exact up to the order of the atomic sums (1e-12)."""
    import paper_2301_02387_gb300 as pkg
    gm, om, op, _, perm = space
    x = np.random.default_rng(0).standard_normal((om.N, 5))
    a, b = _apply(gm, pkg.OP_STIFF, x, perm), _apply(gm, pkg.OP_STIFF, x * 2.0 ** -1000, perm)
    assert_close(b * 2.0 ** 500 * 2.0 ** 500, a, 1e-12, axis=0, what="scaled stiffness")


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_value_stays_on_its_lines(space, value):
    import paper_2301_02387_gb300 as pkg
    gm, om, op, A_abs, perm = space
    x = np.random.default_rng(1).standard_normal((om.N, 2))
    at = np.flatnonzero(op.interior)[om.N // 5]
    x[at, 1] = value
    got = np.empty_like(x)
    got[perm] = _apply(gm, pkg.OP_STIFF, x, perm)
    on = np.asarray(A_abs[:, [at]].todense())[:, 0] > 0
    assert np.isfinite(got[:, 0]).all() and np.isfinite(got[~on, 1]).all()
    assert not np.isfinite(got[on, 1]).any()
    assert np.isnan(got[at, 1]) if np.isnan(value) else got[at, 1] == value
