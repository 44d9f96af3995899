"""GPU: double-float implicit steps whose first refinement rounds come from one shared
Chebyshev expansion, against the same call with an own inner solve per round (max_iter just
below what the expansion needs keeps those) and against the oracle: odd rows and rows a
vector width divides, meshes with one-cell axes, periodic axes, both implicit schemes,
several fields of which one has no mean and one is zero, one run of steps and several
(20 steps to a run), small and large dtau / dx^2.

Tolerance: either path ends every step with ||r|| <= 1e-13 ||b|| and ||A^-1|| = 1, so a
field of n steps is within n 1e-13 of the exact steps in the 2-norm relative to the
largest ||b||, and the two paths within 2 n 1e-13 of each other; times 40 for the largest
cell against the root mean square.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def solve(cg, dims, u, c, nsteps, scheme, period, max_iter=10000):
    import torch
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0, periodic=period)
    x = torch.from_numpy(u).cuda()
    _, rep = cg.diffuse(mesh, x, cg.Params(T=c * nsteps, nsteps=nsteps, scheme=scheme, max_iter=max_iter,
                                           precision=cg.PREC_FP32_DF_REFINE), report=True)
    again = torch.from_numpy(u).cuda()
    cg.diffuse(mesh, again, cg.Params(T=c * nsteps, nsteps=nsteps, scheme=scheme, max_iter=max_iter,
                                      precision=cg.PREC_FP32_DF_REFINE))
    mesh.close()
    assert torch.equal(x, again)          # the same schedule, the same bits
    assert rep["final_rel_residual"] <= 1e-13
    return x.cpu().numpy(), rep


CASES = [((32, 24, 16), 0.1, 10), ((33, 20, 17), 0.225, 10), ((97, 9, 5), 0.05, 21), ((128, 8, 8), 0.4, 5),
         ((132, 10, 9), 0.1, 41), ((1, 37, 20), 0.3, 8), ((20, 1, 1), 0.5, 7), ((64, 48, 40), 1.6, 10),
         ((7, 5, 3), 0.02, 4)]


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("period", [(0, 0, 0), (1, 0, 0), (1, 1, 1)])
@pytest.mark.parametrize("dims,c,nsteps", CASES)
def test_shared_expansion_matches_own_solves(dims, c, nsteps, period, scheme):
    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(n + nsteps)
    u = np.stack([rng.random(n), rng.standard_normal(n), np.zeros(n)])
    got, rep = solve(cg, dims, u, c, nsteps, scheme, period)
    own_m = rep["inner_iters_per_round"]
    cap = own_m - 1 if own_m > 2 else 2
    ref, rep_own = solve(cg, dims, u, c, nsteps, scheme, period, max_iter=cap)
    assert not np.any(got[2])
    for f in (0, 1):
        bound = 2e-13 * nsteps * np.sqrt(np.mean(u[f] ** 2)) * 40
        assert np.max(np.abs(got[f] - ref[f])) <= bound
    if n <= 30_000 and nsteps <= 10:
        import oracle
        exact, _ = oracle.diffuse_structured(u[:2], dims, 1.0, c * nsteps, nsteps, scheme, periodic=period)
        assert np.max(np.abs(got[:2] - exact)) <= 1e-10 * np.max(np.abs(exact))


def test_shared_expansion_saves_applications_and_yields_to_limits():
    """Fewer operator applications than own solves; a workspace limit without room for the
    expansion's vectors falls back to those."""
    import torch

    import paper_1409_0001_gb300 as cg
    dims, n = (64, 64, 64), 64 ** 3
    u = np.random.default_rng(1).random((1, n))
    got, rep = solve(cg, dims, u, 0.1, 10, 0, (0, 0, 0))
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
    x = torch.from_numpy(u).cuda()
    try:
        cg.set_workspace_limit(cg.workspace_bytes() + 14 * 8 * n)
        _, tight = cg.diffuse(mesh, x, cg.Params(T=1.0, nsteps=10, precision=cg.PREC_FP32_DF_REFINE), report=True)
    finally:
        cg.set_workspace_limit(0)
        mesh.close()
    assert rep["iters"] < 0.8 * tight["iters"]
    assert np.max(np.abs(got - x.cpu().numpy())) <= 2e-12 * 40


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("nsteps", [2, 6, 20, 21])
def test_batches_match_single_meshes(nsteps, scheme):
    """Uneven snapshots (odd and single-cell sides, rows over one tile) with bandwidths of
    their own: both schedules give the same bits, and each snapshot what its own call gives
    to the tolerance above (21 steps are more than a batch's one run: own solves)."""
    import torch

    import paper_1409_0001_gb300 as cg
    dims = [(33, 20, 17), (5, 1, 1), (64, 9, 3), (1, 30, 4), (130, 6, 5), (40, 40, 12)]
    cs = [0.1, 0.3, 0.05, 0.2, 0.4, 0.15]
    rng = np.random.default_rng(nsteps)
    us = [np.stack([rng.random(a * b * d), rng.standard_normal(a * b * d)]) for a, b, d in dims]
    bw = [2.0 * np.sqrt(c * nsteps) for c in cs]
    got = {}
    for shape in (4, 504, 516):
        meshes = [cg.StructuredMesh(d, (0, 0, 0), 1.0) for d in dims]
        x = [torch.from_numpy(u).cuda() for u in us]
        _, rep = cg.diffuse_batched(meshes, x, cg.Params(nsteps=nsteps, scheme=scheme, sweep_shape=shape,
                                                         precision=cg.PREC_FP32_DF_REFINE),
                                    bandwidths=bw, report=True)
        assert rep["final_rel_residual"] <= 1e-13
        got[shape] = [t.cpu().numpy() for t in x]
        for m in meshes:
            m.close()
    for s, d in enumerate(dims):
        assert np.array_equal(got[4][s], got[504][s]) and np.array_equal(got[504][s], got[516][s])
        lone, _ = solve(cg, d, us[s], cs[s], nsteps, scheme, (0, 0, 0))
        for f in (0, 1):
            bound = 2e-13 * nsteps * np.sqrt(np.mean(us[s][f] ** 2)) * 40
            assert np.max(np.abs(got[504][s][f] - lone[f])) <= bound


@pytest.mark.parametrize("dims,period", [((32, 24, 16), (0, 0, 0)), ((33, 20, 17), (0, 0, 0)),
                                         ((64, 10, 9), (1, 0, 0)), ((30, 12, 7), (1, 1, 1))])
@pytest.mark.parametrize("scheme", [0, 1])
def test_bf16_inner_storage_takes_the_fp32_increments(dims, period, scheme):
    """BF16 inner storage: the expansion's FP32 increments, then BF16 rounds; against FP32
    storage to the tolerance above.  A round cap below its five own rounds stays refused."""
    import torch

    import paper_1409_0001_gb300 as cg
    n = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(n)
    u = np.stack([rng.random(n), rng.standard_normal(n)])
    ref, _ = solve(cg, dims, u, 0.2, 8, scheme, period)
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0, periodic=period)
    par = dict(T=1.6, nsteps=8, scheme=scheme, precision=cg.PREC_BF16_DF_REFINE)
    x = torch.from_numpy(u).cuda()
    _, rep = cg.diffuse(mesh, x, cg.Params(**par), report=True)
    assert rep["final_rel_residual"] <= 1e-13
    for f in (0, 1):
        assert np.max(np.abs(x[f].cpu().numpy() - ref[f])) <= 2e-13 * 8 * np.sqrt(np.mean(u[f] ** 2)) * 40
    with pytest.raises(cg.CGError):
        cg.diffuse(mesh, torch.from_numpy(u).cuda(), cg.Params(max_rounds=4, **par))
    mesh.close()
