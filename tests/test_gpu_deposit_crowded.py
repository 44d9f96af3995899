"""GPU: ordered depositions with and without a cell of more than 64 particles in turn on one mesh
(radix sort and counting sort; the launches ahead of the host's look at the counters do nothing
where a cell is crowded, and a mesh whose last call was crowded looks first): the oracle's
bits each time, no output on an error in between, and no launch of the counting sort in a
second crowded call.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS = (6, 5, 4)
N = 120
LOCATE, RADIX_PASS, HEADS = 1, 4, 1   # launches; a pass: upsweep, two of the scan, downsweep


def particles(rng, per_cell, nf):
    cell = rng.permutation(np.repeat(np.arange(N), np.resize(per_cell, N)))
    pos = np.stack([cell % 6, cell // 6 % 5, cell // 30]) + rng.random((3, len(cell)))
    return cell.astype(np.int32), pos, rng.standard_normal((nf, len(cell)))


def launches(cg, f):
    lib = cg.load_library()
    lib.cg_launch_count_reset()
    got = f()
    return got, lib.cg_launch_count()


@pytest.mark.parametrize("nf", [1, 3])
def test_crowded_and_not_in_turn(nf):
    import torch

    import oracle
    import paper_1409_0001_gb300 as cg
    rng = np.random.default_rng(nf)
    mesh = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    crowded_before = False
    for per_cell in ([1, 2], [65, 0], [3, 200], [64], [2, 0], [66], [5], [0, 70], [0, 90]):
        cell, pos, w = particles(rng, per_cell, nf)
        ref, _ = oracle.deposit(cell, w, N)
        p, v = torch.from_numpy(pos).cuda(), torch.from_numpy(w).cuda()
        out = torch.full((nf, N), 7.0, dtype=torch.float64, device="cuda")
        bad = p.clone()
        bad[0, -1] = -1.0
        with pytest.raises(cg.CGError):
            cg.deposit(mesh, bad, v, out=out)
        assert bool((out == 7.0).all())
        got, k = launches(cg, lambda: cg.deposit(mesh, p, v, out=out))
        assert np.array_equal(got.cpu().numpy(), ref)
        crowded = max(per_cell) > 64
        if crowded and crowded_before:
            assert k == LOCATE + RADIX_PASS + HEADS
        crowded_before = crowded
    mesh.close()


def test_batch_with_some_crowded():
    import torch

    import oracle
    import paper_1409_0001_gb300 as cg
    rng = np.random.default_rng(9)
    meshes = [cg.StructuredMesh(DIMS, (0, 0, 0), 1.0) for _ in range(3)]
    for counts in (([1], [80], [2]), ([90], [3], [2]), ([4], [5], [70, 0])):
        parts = [particles(rng, c, 2) for c in counts]
        pos = [torch.from_numpy(p).cuda() for _, p, _ in parts]
        w = [torch.from_numpy(v).cuda() for _, _, v in parts]
        par = cg.Params(T=1.0, nsteps=4, precision=3, sweep_shape=504)
        got = cg.coarse_grain_batched(meshes, pos, w, par)
        again = [torch.from_numpy(oracle.deposit(c, v, N)[0]).cuda() for c, _, v in parts]
        cg.diffuse_batched(meshes, again, par)
        assert all(torch.equal(a, b) for a, b in zip(got, again))
    for m in meshes:
        m.close()
