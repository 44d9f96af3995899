"""GPU: the ordered deposition at the edges of its per-cell paths -- cells of 0, 1, 2, 3, 4,
5, 8, 9, 64 and (radix sort) 65 particles, one cell, cell counts around one scan chunk and
around the scan's inline limit, several fields -- bit for bit against the oracle, and no
output written when a particle lies outside or a weight is not finite.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,per_cell,nf", [((4, 3, 2), [0, 1, 2, 3, 4, 5, 8, 9, 64], 1),
                                              ((4, 3, 2), [0, 1, 7, 8, 9, 65], 3), ((1, 1, 1), [5], 2),
                                              ((16, 16, 16), [0, 1, 2, 5], 2), ((4095, 1, 1), [1, 0], 1),
                                              ((256, 256, 128), [0, 0, 1], 1), ((256, 257, 128), [0, 1, 0, 0], 2)])
def test_ordered_sums(dims, per_cell, nf):
    import torch

    import oracle
    import paper_1409_0001_gb300 as cg
    n_cells = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(n_cells)
    count = np.resize(per_cell, n_cells)
    cell = rng.permutation(np.repeat(np.arange(n_cells), count))
    pos = np.stack([cell % dims[0], cell // dims[0] % dims[1], cell // (dims[0] * dims[1])]) + rng.random((3, len(cell)))
    w = rng.standard_normal((nf, len(cell))) * 10.0 ** rng.integers(-8, 8, (nf, len(cell)))
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
    got = cg.deposit(mesh, torch.from_numpy(pos).cuda(), torch.from_numpy(w).cuda()).cpu().numpy()
    ref, _ = oracle.deposit(cell.astype(np.int32), w, n_cells)
    assert np.array_equal(got, ref)
    out = torch.full((nf, n_cells), 7.0, dtype=torch.float64, device="cuda")
    for bad_pos, bad_w in ((True, False), (False, True)):
        p, v = pos.copy(), w.copy()
        if bad_pos:
            p[0, -1] = -1.0
        if bad_w:
            v[-1, 0] = np.inf
        with pytest.raises(cg.CGError):
            cg.deposit(mesh, torch.from_numpy(p).cuda(), torch.from_numpy(v).cuda(), out=out)
        assert bool((out == 7.0).all())
    mesh.close()
