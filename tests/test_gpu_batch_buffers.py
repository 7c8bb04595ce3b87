"""A batch that replays a graph, called with other buffers and other fields: the
second call works on the second call's (an odd orbital count has no instance table,
which is what the buffers used to be looked up in).

Bar 2e-6: both calls are the same float32 passes, up to the order of their atomic sums.
"""
import pytest

pytestmark = pytest.mark.gpu

NUC = [((0.0, 0.0, 0.7), 1.0, 1), ((0.0, 0.0, -0.7), 1.0, 1)]


@pytest.mark.parametrize("counts", [(1, 3), (2, 4), (2, 3)])
def test_new_buffers_and_fields(counts):
    import torch
    import paper_2301_02387_gb300 as pkg
    meshes = [pkg.Mesh(-8.0, 8.0, 4 + i, 2 + i, NUC, 2.0) for i in range(len(counts))]
    batch = pkg.Batch(meshes)

    def call(seed, E, keep):
        g = torch.Generator().manual_seed(seed)
        xs = [torch.randn((m.N, n), generator=g, dtype=torch.complex64).cuda() for m, n in zip(meshes, counts)]
        ys = [torch.full_like(x, float("nan")) for x in xs]
        keep += xs + ys
        batch.apply(pkg.OP_H1_C64, xs, ys, E=E)
        for m, x, y, e in zip(meshes, xs, ys, E):
            ref = pkg.op_apply(m, pkg.OP_H1_C64, x, torch.empty_like(x), E=e)
            assert float((y - ref).norm() / ref.norm()) < 2e-6
        return xs, ys

    keep = []
    xs, ys = call(1, [(0.1, 0.0, 0.0), (0.0, 0.2, 0.0)], keep)
    call(2, [(0.1, 0.0, 0.0), (0.0, 0.2, 0.0)], keep)          # other buffers
    for E in ([(0.3, 0.0, 0.1), (0.0, 0.0, 5.0)], [(0.0, 0.0, 0.0), (0.0, 1.0, 0.0)]):   # other fields, first buffers
        batch.apply(pkg.OP_H1_C64, xs, ys, E=E)
        for m, x, y, e in zip(meshes, xs, ys, E):
            ref = pkg.op_apply(m, pkg.OP_H1_C64, x, torch.empty_like(x), E=e)
            assert float((y - ref).norm() / ref.norm()) < 2e-6
