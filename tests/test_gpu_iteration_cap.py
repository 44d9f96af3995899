"""GPU: the cap on inner iterations (max_iter) of a double-float call holds for that call, whatever
caps earlier calls on the mesh had: status (the smallest cap does not converge), report and bits
as on a fresh mesh.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [3, 4])
def test_caps_in_turn(precision):
    import torch

    import paper_1409_0001_gb300 as cg
    dims = (24, 20, 18)
    u = torch.from_numpy(np.random.default_rng(1).random((1, 24 * 20 * 18))).cuda()
    kept = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
    for cap in (3, 6, 4, 10000, 3):
        got = []
        fresh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
        for mesh in (kept, fresh):
            x = u.clone()
            par = cg.Params(T=2.0, nsteps=5, precision=precision, max_iter=cap, sweep_shape=102)
            try:
                _, rep = cg.diffuse(mesh, x, par, report=True)
                assert rep["inner_iters_per_round"] <= cap
                got.append((x, rep["iters"], rep["refine_rounds"], rep["final_rel_residual"]))
            except cg.CGError as e:
                got.append((x, e.code))
        assert torch.equal(got[0][0], got[1][0]), cap
        assert got[0][1:] == got[1][1:], cap
        fresh.close()
    kept.close()
