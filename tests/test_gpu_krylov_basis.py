"""The integer Gram-Schmidt passes at their edges, through the entry points:
every staging depth (Krylov dimensions around 4, 10 and 14), every orbital count
(threads of a tile left idle when 256 is no multiple of it), columns of very
different size, exact zeros, power-of-two scaling and non-finite input.

Bars: the oracle comparison is the FP64 parity bar of the propagator, 1e-10.
Scaling the start vector by a power of two scales every product exactly, so the
results agree up to the order of the cell pass's float64 atomics, which a
propagation of a few steps amplifies to well below 1e-12.
"""
import numpy as np
import pytest

from oracle import fem, krylov, mctdhf, mesh as omesh
from paper_2301_02387_gb300 import inputs
from tests._match import assert_close, coord_permutation

pytestmark = pytest.mark.gpu

CASE = (-7.0, 7.0, 3, 2, [((0.0, 0.0, 0.7), 1.0, 1), ((0.0, 0.0, -0.7), 1.0, 1)], 2.0)


@pytest.fixture(scope="module")
def space():
    import paper_2301_02387_gb300 as pkg
    gm, om = pkg.Mesh(*CASE), omesh.Mesh(*CASE)
    op = fem.Operators(om)
    return gm, om, op, coord_permutation(gm.tables()[0], om.Xm)


@pytest.mark.parametrize("n,m", [(1, 1), (2, 3), (3, 5), (4, 10), (5, 11), (6, 14), (7, 15), (8, 16)])
@pytest.mark.parametrize("spread", [1.0, 1e-7])
def test_columns_and_dimensions(space, n, m, spread):
    """phi with columns scaled by spread^(p/n): one exponent per group of rows and column."""
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    interior = ~om.boundary
    phi_o = inputs.lowdin(inputs.molecular_orbitals(om.Xm, interior, CASE[4], n), op.ML)
    phi_o = phi_o * spread ** (np.arange(n) / n)
    U_o = np.zeros((n, n, om.N), dtype=np.complex128)
    E = (0.02, -0.01, 0.03)
    sim = mctdhf.MCTDHF.__new__(mctdhf.MCTDHF)
    sim.ops, sim.mesh, sim.n = op, om, n
    sim.interior = interior.astype(np.float64)
    ref, _, _, m_used, _ = krylov.arnoldi_expm(lambda v: sim.G_apply(v, phi_o, U_o, E), phi_o, sim.inner, m, 0.01)
    phi = torch.from_numpy(np.ascontiguousarray(phi_o[perm])).cuda()
    out, _, mu, _ = pkg.arnoldi_step(gm, phi, None, m, 0.01, E=E)
    torch.cuda.synchronize()
    assert mu == m_used
    got = out.cpu().numpy()
    assert_close(got, ref[perm], 1e-10, what="step")
    assert np.all(got[om.boundary[perm]] == 0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("power", [-500, -60])
def test_power_of_two_scaling(space, precision, power):
    """The linear propagator (one orbital, no projector) commutes with a scaling by
    2^power (downwards: the breakdown rule compares h with 1e-14 |phi|, so a start
    vector of norm 2^100 breaks down at once by definition)."""
    import torch
    from paper_2301_02387_gb300 import adjoint as adj
    gm, om, op, perm = space
    if precision and power < -100:   # the complex64 copy of the start vector holds about 2^-126
        power = -60
    phi_o = inputs.lowdin(inputs.molecular_orbitals(om.Xm, ~om.boundary, CASE[4], 1), op.ML)[:, 0]
    phi = torch.from_numpy(np.ascontiguousarray(phi_o[perm])).cuda()
    Ek = np.array([0.03, -0.02])
    args = dict(dt=0.01, krylov_m=9, tol=1e-10, precision=precision, want_end=True)
    _, a, _ = adj.tdse_forward(gm, phi, Ek, **args)
    _, b, _ = adj.tdse_forward(gm, phi * 2.0 ** power, Ek, **args)
    bar = 1e-6 if precision else 1e-12
    assert_close((b * 2.0 ** -power).cpu().numpy(), a.cpu().numpy(), bar, what="scaled propagation")


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("precision", [0, 1])
def test_non_finite_input_is_reported(space, value, precision):
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    phi_o = inputs.lowdin(inputs.molecular_orbitals(om.Xm, ~om.boundary, CASE[4], 2), op.ML)
    phi = torch.from_numpy(np.ascontiguousarray(phi_o[perm])).cuda()
    phi[gm.n_interior // 2, 1] = value
    with pytest.raises(pkg.AfemError):
        pkg.arnoldi_step(gm, phi, None, 6, 0.01, precision=precision)


def test_zero_column(space):
    """A column that is exactly zero stays zero (its groups carry no exponent)."""
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    phi_o = inputs.lowdin(inputs.molecular_orbitals(om.Xm, ~om.boundary, CASE[4], 2), op.ML)
    phi_o[:, 1] = 0
    phi = torch.from_numpy(np.ascontiguousarray(phi_o[perm])).cuda()
    out = pkg.arnoldi_propagate(gm, phi, None, 8, 0.02, 1e-10)[0]
    assert torch.all(out[:, 1] == 0) and torch.isfinite(torch.view_as_real(out)).all()
