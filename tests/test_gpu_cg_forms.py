"""GPU: the two forms of the FP64 conjugate gradients -- one cooperative launch where the
mesh fits in the SMs' registers, and two launches per iteration beyond that or where its
workspace is refused -- against the oracle and against each other, at sizes around their
edges: fewer cells than a block, one cell per thread and one more, remainders, one-cell
axes, periodic axes, several fields, both implicit schemes.

Tolerance: both stop at ||r|| <= 1e-13 ||b|| per step, so each is within a few 1e-13 of the
exact steps (times at most 1 + 12 dtau/dx^2 = 4 here, through ten steps): 1e-11 covers the
difference of two such runs with a margin of ten, 1e-10 is the FP64 bar of the oracle.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS = [(1, 1, 1), (5, 1, 1), (7, 3, 2), (33, 8, 9), (64, 32, 38), (77, 32, 32), (96, 97, 100), (100, 97, 96),
        (101, 99, 98)]


def solve(cg, dims, u, nf, scheme, period=(0, 0, 0), limit=0):
    import torch
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 0.5, periodic=period)
    x = torch.from_numpy(u).cuda()
    try:
        if limit:
            cg.set_workspace_limit(cg.workspace_bytes() + limit)
        _, rep = cg.diffuse(mesh, x, cg.Params(T=0.25 * 0.25 * 5, nsteps=5, scheme=scheme), report=True)
    finally:
        cg.set_workspace_limit(0)
        mesh.close()
    return x.cpu().numpy(), rep


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("scheme", [0, 1])
def test_forms_match_oracle(dims, scheme):
    import oracle
    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    u = np.random.default_rng(n).random((1, n))
    got, rep = solve(cg, dims, u, 1, scheme)
    assert rep["final_rel_residual"] <= 1e-13
    if n <= 50_000:
        ref, _ = oracle.diffuse_structured(u, dims, 0.5, 0.25 * 0.25 * 5, 5, scheme)
        assert np.max(np.abs(got - ref)) <= 1e-10 * np.max(np.abs(ref))
    else:   # too large for the oracle here: against the double-float solver
        import torch
        mesh = cg.StructuredMesh(dims, (0, 0, 0), 0.5)
        x = torch.from_numpy(u).cuda()
        cg.diffuse(mesh, x, cg.Params(T=0.25 * 0.25 * 5, nsteps=5, scheme=scheme,
                                      precision=cg.PREC_FP32_DF_REFINE))
        assert np.max(np.abs(got - x.cpu().numpy())) <= 1e-11 * np.max(np.abs(got))
        mesh.close()


@pytest.mark.parametrize("dims", [(33, 8, 9), (96, 97, 100)])
@pytest.mark.parametrize("period", [(0, 0, 0), (1, 0, 0), (0, 1, 1), (1, 1, 1)])
def test_forms_match_each_other(dims, period):
    """Four fields at once (one of them zero, one constant) against one field alone."""
    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(7)
    u = np.stack([rng.random(n), rng.standard_normal(n), np.zeros(n), np.full(n, 3.0)])
    got, rep = solve(cg, dims, u, 4, 0, period)
    assert np.array_equal(got[2], u[2])
    lone, rep1 = solve(cg, dims, u[:1], 1, 0, period)
    assert np.max(np.abs(lone[0] - got[0])) <= 1e-11 * np.max(np.abs(got[0]))
    assert rep["iters"] >= rep1["iters"]


def test_two_launch_form_under_a_workspace_limit():
    """A limit that holds three vectors of a mesh beyond the cooperative form, not four: the
    call runs and gives what the unlimited one gives."""
    import paper_1409_0001_gb300 as cg
    dims = (101, 99, 98)
    n = dims[0] * dims[1] * dims[2]
    u = np.random.default_rng(3).random((1, n))
    full, _ = solve(cg, dims, u, 1, 0)
    tight, _ = solve(cg, dims, u, 1, 0, limit=int(3 * 8 * n * 1.2))
    assert np.max(np.abs(full - tight)) <= 1e-11 * np.max(np.abs(full))
