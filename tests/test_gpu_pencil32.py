"""The float32 line-sweep form of the stiffness and of H1~: lane groups of 4, 2
and 1 floats (by count and by alignment), counts around the 16 floats of a
block, the last block's fewer cells, against the oracle's assembled matrices.
Bar 2e-5 per column, the float32 parity bar of the operators; surface entries
of x may hold anything in the masked operator."""
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


def _apply(gm, kind, x_host, offset, E=None):
    """The operator on buffers `offset` floats behind a 16-byte boundary."""
    import torch
    import paper_2301_02387_gb300 as pkg
    cplx = np.iscomplexobj(x_host)
    f = np.ascontiguousarray(x_host.astype(np.complex64 if cplx else np.float32))
    flat = torch.zeros(f.view(np.float32).size + 4, dtype=torch.float32, device="cuda")
    out = torch.zeros_like(flat)
    n = f.view(np.float32).size
    flat[offset:offset + n] = torch.from_numpy(f.view(np.float32).reshape(-1)).cuda()
    if cplx:
        x = torch.view_as_complex(flat[offset:offset + n].view(-1, 2)).view(f.shape)
        y = torch.view_as_complex(out[offset:offset + n].view(-1, 2)).view(f.shape)
    else:
        x, y = flat[offset:offset + n].view(f.shape), out[offset:offset + n].view(f.shape)
    pkg.op_apply(gm, kind, x, y, E=E)
    assert float(out[:offset].abs().sum()) == 0.0 and float(out[offset + n:].abs().sum()) == 0.0
    return y.cpu().numpy()


@pytest.mark.parametrize("k", [1, 2, 4, 9, 16, 18, 20, 36, 64])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_stiffness(space, k, offset):
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    x = np.random.default_rng(k).standard_normal((om.N, k))
    got = _apply(gm, pkg.OP_STIFF_F32, x[perm], offset)
    assert_close(got, op.stiffness_apply(x)[perm], 2e-5, axis=0, what="stiffness")


@pytest.mark.parametrize("n", [1, 2, 3, 5, 8, 9, 13])
@pytest.mark.parametrize("offset", [0, 2])
def test_h1(space, n, offset):
    import paper_2301_02387_gb300 as pkg
    gm, om, op, perm = space
    rng = np.random.default_rng(n)
    x = rng.standard_normal((om.N, n)) + 1j * rng.standard_normal((om.N, n))
    ref = op.h1_apply(x, E=(0.05, -0.02, 0.1))[perm]
    xs = x[perm].copy()
    xs[gm.n_interior:] = np.nan
    got = _apply(gm, pkg.OP_H1_C64, xs, offset, E=(0.05, -0.02, 0.1))
    assert_close(got, ref, 2e-5, axis=0, what="H1")
