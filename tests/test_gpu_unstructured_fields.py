"""GPU: the unstructured Chebyshev passes on field counts around their group of four (one
field has a kernel of its own) and on cell counts around a block's pass of 512 cells:
several fields at once against each field alone.

Tolerance: either run ends every step with ||r|| <= 1e-13 ||b||; the scaled operator's
inverse is at most 1 in the mass norm, so two runs of n = 6 steps differ by at most
2 n 1e-13 of the field's norm, times 40 for the largest cell and 20 for the ratio of the
largest to the smallest cell volume.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,size", [("tet", 3), ("tet", 5), ("tet", 8), ("hex", 3), ("hex", 8), ("hex", 33)])
@pytest.mark.parametrize("nf", [2, 4, 5, 9])
def test_fields_together_and_alone(kind, size, nf):
    import torch

    import paper_1409_0001_gb300 as cg
    import workloads as W
    if kind == "tet":
        mesh = cg.TetMesh(*W.kuhn_tet_mesh(size, jitter=0.1))
    else:
        f = np.cumsum(np.concatenate([[0.0], 1.03 ** np.arange(size)]))
        mesh = cg.HexMesh(np.linspace(0, 1, size + 1), np.linspace(0, 1, size + 2), f / f[-1])
    u = np.random.default_rng(size).random((nf, mesh.ncells))
    p = cg.Params(bandwidth=2.0 / size, nsteps=6, precision=cg.PREC_FP32_REFINE)
    x = torch.from_numpy(u).cuda()
    _, rep = cg.diffuse(mesh, x, p, report=True)
    assert rep["final_rel_residual"] <= 1e-13
    for q in range(nf):
        y = torch.from_numpy(u[q:q + 1]).cuda()
        cg.diffuse(mesh, y, p)
        bound = 2 * 6 * 1e-13 * 40 * 20 * np.sqrt(np.mean(u[q] ** 2))
        assert float((x[q] - y[0]).abs().max()) <= bound
    mesh.close()
