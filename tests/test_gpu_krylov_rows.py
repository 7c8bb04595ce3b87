"""The integer Gram-Schmidt passes with several rows per thread and several tiles
per block (meshes of 50,653 to 132,651 points: 2 and 4 rows, up to two tiles),
rings of every depth, entry by entry on orbitals that fall by 2^20 from node to
node, so that the rows of one thread differ by far more than float64 holds.

Bars: an entry of the oracle's float64 propagation follows from the entries around
it, a few hundred roundings (1e-13); 1e-8 of the entry leaves room for entries in
which these cancel.  Norms: 1e-10 and 1e-6, the parity bars of the two forms.
"""
import functools

import numpy as np
import pytest

from oracle import fem, krylov, mctdhf, mesh as omesh
from tests._match import coord_permutation

pytestmark = pytest.mark.gpu

CASES = [(36, 8, 2), (36, 8, 11), (36, 7, 15), (36, 7, 16), (50, 3, 3), (50, 3, 15), (43, 1, 11)]   # cells per axis, orbitals, m


@functools.lru_cache(maxsize=2)
def _space(nc):
    import paper_2301_02387_gb300 as pkg
    case = (-0.5 * nc, 0.5 * nc, nc, 1, [((0.2, 0.1, 0.3), 1.0, 0)], 2.0)
    gm, om = pkg.Mesh(*case), omesh.Mesh(*case)
    return gm, om, fem.Operators(om), coord_permutation(gm.tables()[0], om.Xm)


def _orbitals(om, n, step):
    """Column j falls by 2^-step from node to node away from a node of its own (zero below 2^-700)."""
    rng = np.random.default_rng(n)
    X, phi = np.round(om.Xm - om.Xm.min(0)), np.empty((om.N, n), dtype=np.complex128)
    for j in range(n):
        d = np.abs(X - np.round(X.max(0) / 2 + rng.integers(-4, 5, 3))).sum(1)
        phi[:, j] = np.where(step * d < 700, 2.0 ** -np.minimum(step * d, 700), 0.0) * np.exp(2j * np.pi * rng.random(om.N))
    phi[om.boundary] = 0
    return phi


def _reference(om, op, phi, m, dt, shift):
    sim = mctdhf.MCTDHF.__new__(mctdhf.MCTDHF)
    n = phi.shape[1]
    sim.ops, sim.mesh, sim.n = op, om, n
    sim.interior = (~om.boundary).astype(np.float64)
    U = np.zeros((n, n, om.N), dtype=np.complex128)
    for j in range(n):
        U[j, j] = shift
    E = (0.02, -0.01, 0.03)
    return krylov.arnoldi_expm(lambda v: sim.G_apply(v, phi, U, E), phi, sim.inner, m, dt)[0], E


@pytest.mark.parametrize("shift", [0.0, 3e3])   # a large shift calls for the second Gram-Schmidt pass
@pytest.mark.parametrize("nc,n,m", CASES)
def test_against_the_oracle_entry_by_entry(nc, n, m, shift):
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = _space(nc)
    phi_o = _orbitals(om, n, 20)
    dt = 0.1 / (1.0 + shift)
    ref, E = _reference(om, op, phi_o, m, dt, shift)
    ref = ref[perm]
    phi = torch.from_numpy(np.ascontiguousarray(phi_o[perm])).cuda()
    U = None
    if shift:
        U = (shift * torch.eye(n, dtype=torch.complex128, device="cuda")).expand(gm.N, n, n).contiguous()
    for precision, bar in ((0, 1e-10), (1, 1e-6)):
        out = pkg.arnoldi_step(gm, phi, U, m, dt, E=E, precision=precision)[0].cpu().numpy()
        assert np.linalg.norm(out - ref) <= bar * np.linalg.norm(ref)
        if precision == 0 and shift == 0.0 and m <= 11:   # (a shift cancels in the entries; the
            # exponential's Taylor polynomial has the last coefficients of larger m in norm only)
            big = np.abs(ref) > 2.0 ** -600
            assert np.all(np.abs(out - ref)[big] <= 1e-8 * np.abs(ref)[big])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nc,n", [(36, 8), (36, 7), (50, 3), (43, 1)])
def test_one_vector_is_a_phase(nc, n, precision):
    """m = 1: phi times one number (of modulus 1 in FP64), in every entry to a few roundings."""
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = _space(nc)
    phi_o = _orbitals(om, n, 7)[perm]
    out = pkg.arnoldi_step(gm, torch.from_numpy(phi_o).cuda(), None, 1, 0.01, E=(0.1, 0.0, 0.0), precision=precision)[0]
    out, at = out.cpu().numpy(), np.argmax(np.abs(phi_o))
    ratio = out.flat[at] / phi_o.flat[at]
    if precision == 0:   # (the complex64 cell pass leaves h_00 an imaginary part)
        assert abs(abs(ratio) - 1.0) < 1e-13
    assert np.all(np.abs(out - ratio * phi_o) <= 1e-14 * np.abs(phi_o))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("value", [0.0, np.nan, np.inf])
def test_zero_columns_and_non_finite_entries(value, precision):
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = _space(36)
    phi = torch.from_numpy(_orbitals(om, 8, 1)[perm]).cuda()
    if value == 0.0:
        phi[:, 3] = 0
        out = pkg.arnoldi_step(gm, phi, None, 6, 0.01, precision=precision)[0]
        assert torch.all(out[:, 3] == 0) and torch.isfinite(torch.view_as_real(out)).all()
    else:
        phi[gm.n_interior // 2, 3] = value
        with pytest.raises(pkg.AfemError):
            pkg.arnoldi_step(gm, phi, None, 6, 0.01, precision=precision)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("value", [1e30, np.inf, np.nan])
def test_surface_rows_may_hold_anything(value, precision):
    """The orbitals vanish on the surface: what its rows hold has no part in the result inside
    (two propagations of the same orbitals differ by the order of the scatter's additions)."""
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = _space(36)
    phi = torch.from_numpy(_orbitals(om, 7, 1)[perm]).cuda()
    a = pkg.arnoldi_step(gm, phi, None, 6, 0.01, precision=precision)[0][:gm.n_interior].clone()
    phi[gm.n_interior:] = value
    b = pkg.arnoldi_step(gm, phi, None, 6, 0.01, precision=precision)[0][:gm.n_interior]
    assert float((a - b).norm() / a.norm()) < (1e-13, 1e-6)[precision]
