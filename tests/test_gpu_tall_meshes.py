"""GPU: double-float implicit steps on meshes of very many planes, where a launch of few planes a
block would have more than 65,535 chunks times fields along a grid's z axis, with a stated deep
sweep (the autotuner times shallow ones too, which such meshes have no grid for): several fields
and odd rows, on both sides of the limit.
Against FP64 conjugate gradients to the sum of both stopping tolerances (1e-13 per step
relative to ||b||, five steps) times 100 for the largest cell against the root mean square.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nf,shape", [((4, 4, 131070), 1, 116), ((4, 4, 131072), 1, 116), ((8, 2, 140001), 1, 104),
                                           ((4, 2, 70000), 2, 108), ((3, 3, 262145), 1, -64), ((5, 2, 90000), 3, 8)])
def test_tall(dims, nf, shape):
    import torch

    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    u = np.random.default_rng(n).random((nf, n))
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
    got, ref = torch.from_numpy(u).cuda(), torch.from_numpy(u).cuda()
    _, rep = cg.diffuse(mesh, got, cg.Params(T=1.0, nsteps=5, precision=cg.PREC_FP32_DF_REFINE, sweep_shape=shape),
                        report=True)
    cg.diffuse(mesh, ref, cg.Params(T=1.0, nsteps=5))
    assert rep["final_rel_residual"] <= 1e-13
    assert float((got - ref).abs().max()) <= 100 * 5 * 2e-13
    mesh.close()
