"""Column counts that the other tests leave out: 49 real columns (seven orbitals) at
degree 4, past three blocks of 16 columns, in the stiffness and in whole mean-field
solves by both solvers, and CG reductions with two blocks per SM (36 columns on
about 80,000 interior rows, on 148 to 152 SMs).

Bars: 1e-10 per column, the FP64 parity bar; a solve's residual in the oracle's
matrices 2e-10 for rtol 1e-10; a column alone and among others, both to rtol 1e-10,
within the condition number (< 1e4) times that.
"""
import numpy as np
import pytest

from oracle import fem, mesh as omesh, poisson
from tests._match import assert_close, coord_permutation

pytestmark = pytest.mark.gpu

CASE = (-8.0, 8.0, 3, 4, [((0.3, -0.45, 0.7), 1.0, 2), ((-1.1, 0.2, -0.35), 2.0, 1)], 1.5)


def _orbitals(X, interior, n, seed):
    rng = np.random.default_rng(seed)
    phi = np.stack([np.exp(-0.4 * ((X - rng.standard_normal(3)) ** 2).sum(1)) * np.exp(1j * X @ rng.standard_normal(3))
                    for _ in range(n)], 1)
    phi[~interior] = 0
    return phi


@pytest.fixture(scope="module")
def space():
    import paper_2301_02387_gb300 as pkg
    gm, om = pkg.Mesh(*CASE), omesh.Mesh(*CASE)
    return gm, om, fem.Operators(om), coord_permutation(gm.tables()[0], om.Xm)


@pytest.mark.parametrize("k", [49, 50])
def test_stiffness(space, k):
    import torch
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    x = np.random.default_rng(k).standard_normal((om.N, k))
    X = torch.from_numpy(np.ascontiguousarray(x[perm])).cuda()
    Y = torch.empty_like(X)
    pkg.op_apply(gm, pkg.OP_STIFF, X, Y)
    assert_close(Y.cpu().numpy(), op.stiffness_apply(x)[perm], 1e-10, axis=0, what="stiffness")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("multigrid", [False, True])
def test_mean_fields_of_seven_orbitals(space, precision, multigrid):
    import torch
    import paper_2301_02387_gb300 as pkg
    _, om, op, perm = space
    gm = pkg.Mesh(*CASE)
    if multigrid:
        pkg.mesh_set_option(gm, pkg.OPT_POISSON_SOLVER, pkg.POISSON_MULTIGRID)
    phi_o = _orbitals(om.Xm, ~om.boundary, 7, 3)
    phi = torch.from_numpy(np.ascontiguousarray(phi_o[perm])).cuda()
    W = torch.zeros((gm.N, 49), dtype=torch.float64, device="cuda")
    _, rel, rc = pkg.poisson_batch(gm, phi, W, rtol=1e-10, precision=precision)
    assert rc == 0 and np.all(rel <= 1e-10)
    Wg = np.empty((om.N, 49))
    Wg[perm] = W.cpu().numpy()
    assert np.all(poisson.PoissonSolver(op).residual(Wg, poisson.pair_densities(op, phi_o)[0]) < 2e-10)


def test_two_blocks_per_multiprocessor():
    import torch
    import paper_2301_02387_gb300 as pkg
    gm = pkg.Mesh(-9.0, 9.0, 22, 2, [((0.1, 0.0, 0.3), 1.0, 1)], 1.0)
    X, _, _ = gm.tables()
    assert 2 <= gm.n_interior // (32 * 7 * 152) and gm.n_interior // (32 * 7 * 148) < 3
    phi = torch.from_numpy(_orbitals(X, np.arange(gm.N) < gm.n_interior, 6, 5)).cuda()
    W = torch.zeros((gm.N, 36), dtype=torch.float64, device="cuda")
    _, rel, rc = pkg.poisson_batch(gm, phi, W, rtol=1e-10)
    assert rc == 0 and rel.max() <= 1e-10
    one = torch.zeros((gm.N, 1), dtype=torch.float64, device="cuda")
    pkg.poisson_batch(gm, phi[:, 5:6].contiguous(), one, rtol=1e-10)
    assert float((W[:, 5] - one[:, 0]).norm() / one.norm()) < 1e-6
