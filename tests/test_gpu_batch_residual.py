"""GPU: a batch's steps with the shared expansion are solved as far as a single mesh's: the worst
residual of a batch of one mesh is at most twice the one of its own call.  Both run the
estimated iterations (a batch one more where the count is odd); two iterations fewer leave
1 / sg^2 = 6 to 26 times the residual here (sg = (sqrt(lmax) - 1) / (sqrt(lmax) + 1) 0.41 at
dtau / dx^2 = 0.4, 0.19 at 0.1), the rounding of the same residual in another order far less
than twice.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [0.1, 0.225, 0.4])
@pytest.mark.parametrize("dims", [(48, 48, 48), (64, 40, 36)])
def test_residual_as_in_a_single_call(dims, c):
    import torch

    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    u = torch.from_numpy(np.random.default_rng(n).standard_normal((3, n))).cuda()   # (no mean to hide behind)
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
    x, y = u.clone(), u.clone()
    _, one = cg.diffuse(mesh, x, cg.Params(T=10 * c, nsteps=10, precision=3), report=True)
    _, batch = cg.diffuse_batched([mesh], [y], cg.Params(T=10 * c, nsteps=10, precision=3), report=True)
    assert batch["final_rel_residual"] <= 2 * one["final_rel_residual"]
    mesh.close()
