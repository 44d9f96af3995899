"""Blocked explicit steps on rows of whole vectors (nx % 4 == 0) at the sizes where the
unrolled z march and its tiles change form: fewer planes than the march is unrolled by,
one plane, z chunks and x and y tiles that end on, before and after a tile's edge, walls
and periodic axes.  Against the FP64 oracle's explicit steps.

Bar: a step rounds each value about eight times at relative 2^-24 in values that the step
averages, so nsteps steps stay within 8 nsteps 2^-24 of the largest value: 5.3e-6 for 11
steps.  Every fused_k gives the same bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NSTEPS = 11
BAR = 8 * NSTEPS * 2.0 ** -24


@pytest.fixture(scope="module")
def cg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1409_0001_gb300 as cg
    from paper_1409_0001_gb300 import build
    build.build()
    cg.load_library()
    return cg


@pytest.mark.parametrize("dims", [(4, 1, 1), (8, 32, 1), (12, 33, 2), (120, 26, 3), (124, 27, 4), (128, 32, 5),
                                  (132, 58, 6), (248, 59, 7), (252, 24, 30)])
@pytest.mark.parametrize("periodic", [(False,) * 3, (True, False, False), (False, True, True)])
def test_explicit_tile_edges(cg, orc, dims, periodic):
    import torch
    rng = np.random.default_rng(sum(dims))
    u0 = rng.random((2, int(np.prod(dims)))) - 0.25
    dx = 0.05
    T = 0.16 * dx * dx * NSTEPS
    ref, _ = orc.diffuse_structured(u0, dims, dx, T, NSTEPS, scheme=2, periodic=periodic)
    mesh = cg.StructuredMesh(dims, (0, 0, 0), dx, periodic=periodic)
    first = None
    for k in (1, 2, 3, 4):
        u = torch.from_numpy(u0.copy()).cuda()
        cg.diffuse(mesh, u, cg.Params(T=T, nsteps=NSTEPS, scheme=2, fused_k=k))
        got = u.cpu().numpy()
        assert np.max(np.abs(got - ref)) <= BAR * np.max(np.abs(u0)), k
        first = got if first is None else first
        assert np.array_equal(got.view(np.int64), first.view(np.int64)), k
    mesh.close()
