"""GPU: a batch repeated on the same meshes with other bandwidths gives what fresh meshes give,
bit for bit: its captured launches hold addresses in the batch's arena, whose parts differ in
length with the bandwidths (the Chebyshev weights of all snapshots, the expansions'
coefficients), while the largest bandwidth, and with it the launch counts, stays the same.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [4, 508])
@pytest.mark.parametrize("precision,nsteps", [(3, 4), (3, 24), (4, 4)])
def test_other_bandwidths_on_the_same_meshes(precision, nsteps, shape):
    import torch

    import paper_1409_0001_gb300 as cg
    rng = np.random.default_rng(5)
    dims = [(int(a), int(b), int(c)) for a, b, c in rng.integers(3, 20, (40, 3))]
    us = [rng.random((2, a * b * c)) for a, b, c in dims]
    par = cg.Params(nsteps=nsteps, precision=precision, sweep_shape=shape)

    def run(meshes, b):
        x = [torch.from_numpy(u).cuda() for u in us]
        bw = [b] * len(dims)
        bw[0] = 4.0                       # the most iterations and the longest expansion
        cg.diffuse_batched(meshes, x, par, bandwidths=bw)
        return x

    kept = [cg.StructuredMesh(d, (0, 0, 0), 1.0) for d in dims]
    # the weights' length moves by about 40 (m(3) - m(2)) floats, several 256-byte units
    for b in (3.0, 2.0, 1.0, 3.0):
        got = run(kept, b)
        fresh = [cg.StructuredMesh(d, (0, 0, 0), 1.0) for d in dims]
        ref = run(fresh, b)
        for s in range(len(dims)):
            assert torch.equal(got[s], ref[s]), (b, s)
        for m in fresh:
            m.close()
    for m in kept:
        m.close()
