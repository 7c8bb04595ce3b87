"""The float64 CG reductions at each of their block counts (one to four per SM,
by the rows a thread takes) and with ragged last rows: the mean field of one
orbital's own density, solved alone (one column) and among n^2 columns.

Both solves meet rtol 1e-10 on the same system, so the fields agree to its
condition number (< 1e4 here) times that: 1e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,p", [(3, 2), (24, 2), (17, 3)])
@pytest.mark.parametrize("n", [2, 4, 6, 8])
def test_columns_alone_and_together(nc, p, n):
    import torch
    import paper_2301_02387_gb300 as pkg
    gm = pkg.Mesh(-9.0, 9.0, nc, p, [((0.1, 0.0, 0.3), 1.0, 1)], 1.0)
    X, _, _ = gm.tables()
    rng = np.random.default_rng(nc + n)
    phi = np.stack([np.exp(-0.4 * ((X - rng.standard_normal(3)) ** 2).sum(1)) * np.exp(1j * X @ rng.standard_normal(3))
                    for _ in range(n)], 1)
    phi[gm.n_interior:] = 0
    phi = torch.from_numpy(np.ascontiguousarray(phi)).cuda()
    W = torch.zeros((gm.N, n * n), dtype=torch.float64, device="cuda")
    _, rel, rc = pkg.poisson_batch(gm, phi, W, rtol=1e-10)
    assert rc == 0 and rel.max() <= 1e-10
    for q in (0, n - 1):
        one = torch.zeros((gm.N, 1), dtype=torch.float64, device="cuda")
        _, rel, rc = pkg.poisson_batch(gm, phi[:, q:q + 1].contiguous(), one, rtol=1e-10)
        assert rc == 0 and rel.max() <= 1e-10
        assert float((W[:, q] - one[:, 0]).norm() / one.norm()) < 1e-6
