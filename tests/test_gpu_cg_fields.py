"""GPU: several fields in one FP64 conjugate gradient call.  In the cooperative form fields run in
groups of blocks side by side (one after another on larger meshes), and a field's block layout
does not depend on how many there are: each field has the bits of its own call -- fewer fields
than groups, as many, one more, several turns -- also where a call stops short (all fields after
the same step).  Where the many fields take the two-launch form the results agree to the stopping tolerance: 1e-13 of ||b|| per step
and form, four steps, times 100 for the largest cell against the root mean square.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(d, nf) for d in [(3, 2, 1), (8, 8, 8), (16, 15, 17), (33, 30, 32), (42, 40, 41)] for nf in (2, 3, 5, 9)]
CASES += [((49, 48, 47), 2), ((49, 48, 47), 3), ((64, 64, 63), 5), ((77, 90, 80), 2), ((77, 90, 80), 9)]


def solve(cg, u, dims, **kw):
    import torch
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
    x = torch.from_numpy(u).cuda()
    code = "CG_OK"
    try:
        cg.diffuse(mesh, x, cg.Params(T=2.0, nsteps=4, **kw))
    except cg.CGError as e:
        code = e.code
    mesh.close()
    return x.cpu().numpy(), code


@pytest.mark.parametrize("dims,nf", CASES)
def test_each_field_as_alone(dims, nf):
    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(n + nf)
    u = rng.standard_normal((nf, n))
    u[nf - 1] = 2.5                         # converged from the start, in the last group
    got, code = solve(cg, u, dims, scheme=nf % 2)
    assert code == "CG_OK"
    for f in range(nf):
        lone, _ = solve(cg, u[f:f + 1], dims, scheme=nf % 2)
        assert np.array_equal(got[f], lone[0]), f


@pytest.mark.parametrize("dims", [(8, 8, 8), (33, 30, 32)])
@pytest.mark.parametrize("nf", [4, 6])
def test_no_convergence_stops_every_field_after_the_step(dims, nf):
    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    u = np.random.default_rng(n).standard_normal((nf, n))
    u[0] = 1.0                              # never fails by itself
    got, code = solve(cg, u, dims, max_iter=8)
    assert code == "CG_ENOCONV"
    for f in range(1, nf):
        lone, code = solve(cg, u[f:f + 1], dims, max_iter=8)
        assert code == "CG_ENOCONV"
        assert np.array_equal(got[f], lone[0]), f
    assert np.array_equal(got[0], u[0])


@pytest.mark.parametrize("dims,nf", [((16, 16, 16), 64), ((32, 32, 32), 40), ((49, 48, 47), 9), ((64, 64, 63), 9)])
def test_many_fields(dims, nf):
    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    u = np.random.default_rng(n).standard_normal((nf, n))
    got, code = solve(cg, u, dims)
    assert code == "CG_OK"
    for f in (0, nf // 2, nf - 1):
        lone, _ = solve(cg, u[f:f + 1], dims)
        assert np.max(np.abs(got[f] - lone[0])) <= 100 * 4 * 2e-13
