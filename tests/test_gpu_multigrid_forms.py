"""The multigrid V-cycle in each of its forms: degree pairs 4-2-1, 3-1, 2-1 and
1-1, packed and single columns (n = 1..4: 1, 4, 9 and 16 columns), the coarsest
grid in one block (1, 8 or 16 nodes a thread) and outside it (more interior
nodes than a block takes: the cell passes), and W at an 8-byte address.

The residual the solver reports is the float64 residual of the full system, so
meeting rtol 1e-10 is the check of the operator; the V-cycle is a fixed
preconditioner of CG, so a wrong transfer or coarse solve shows as iterations:
a sound hierarchy takes 9-20 on these meshes, the bar is 40.  Against the
Jacobi-preconditioned solve the fields agree to the condition number (< 1e4
here) times rtol: 1e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# box, coarse cells, degree, levels
MESHES = [(6.0, 3, 4, 1), (6.0, 3, 3, 2), (6.0, 4, 2, 2), (6.0, 5, 1, 2), (10.0, 13, 2, 1), (10.0, 21, 1, 1), (10.0, 24, 1, 1),
          (10.0, 28, 1, 1)]


@pytest.mark.parametrize("box,nc,p,levels", MESHES)
@pytest.mark.parametrize("n", [1, 2, 3, 4])
@pytest.mark.parametrize("precision", [0, 1])
def test_solve(box, nc, p, levels, n, precision):
    import torch
    import paper_2301_02387_gb300 as pkg
    gm = pkg.Mesh(-box, box, nc, p, [((0.1, 0.0, 0.3), 1.0, levels)], 1.0)
    X, _, _ = gm.tables()
    rng = np.random.default_rng(n)
    phi = np.stack([np.exp(-0.4 * ((X - rng.standard_normal(3)) ** 2).sum(1)) * np.exp(1j * X @ rng.standard_normal(3))
                    for _ in range(n)], 1)
    phi[gm.n_interior:] = 0
    phi = torch.from_numpy(np.ascontiguousarray(phi)).cuda()
    ref = torch.zeros((gm.N, n * n), dtype=torch.float64, device="cuda")
    pkg.poisson_batch(gm, phi, ref, rtol=1e-10, precision=precision)
    pkg.mesh_set_option(gm, pkg.OPT_POISSON_SOLVER, pkg.POISSON_MULTIGRID)
    flat = torch.zeros(gm.N * n * n + 1, dtype=torch.float64, device="cuda")
    for W in (flat[:-1].view(gm.N, n * n), flat[1:].view(gm.N, n * n)):   # 16- and 8-byte aligned
        W.zero_()
        it, rel, rc = pkg.poisson_batch(gm, phi, W, rtol=1e-10, precision=precision)
        assert rc == 0 and rel.max() <= 1e-10 and 0 < it <= 40
        assert float((W - ref).norm() / ref.norm()) < 1e-6
