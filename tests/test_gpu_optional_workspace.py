"""GPU: memory that a call can do without (the shared expansion's vectors, A p of the FP64 solver)
never costs another call, or its own, the memory it needs: meshes and repeated calls under a
workspace limit that holds the needed vectors of all of them.  What a call needs is measured
by calls that cannot take more (an iteration cap below what the expansion needs).

Tolerance: with and without the optional vectors every step ends at 1e-13 ||b||, so the results
of n steps differ by at most 2e-13 n in the 2-norm relative to the largest ||b||; times 40 for
the largest cell against the root mean square.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS, NSTEPS = (96, 80, 72), 10
N = DIMS[0] * DIMS[1] * DIMS[2]
CAP = 4            # inner iterations a round: own solves, more rounds of them


@pytest.fixture
def cg():
    import paper_1409_0001_gb300 as cg
    yield cg
    cg.set_workspace_limit(0)


def field(seed):
    import torch
    return torch.from_numpy(np.random.default_rng(seed).random((1, N))).cuda()


def smooth(cg, mesh, u, **kw):
    x = u.clone()
    _, rep = cg.diffuse(mesh, x, cg.Params(T=2.0, nsteps=NSTEPS, precision=3, **kw), report=True)
    assert rep["final_rel_residual"] <= 1e-13
    return x, rep


def near(a, b, u):
    return float((a - b).abs().max()) <= 40 * 2e-13 * NSTEPS * float(u.square().mean().sqrt())


def needed(cg):
    """Workspace of one call that takes no optional vectors."""
    before = cg.workspace_bytes()
    mesh = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    smooth(cg, mesh, field(0), max_iter=CAP)
    got = cg.workspace_bytes() - before
    mesh.close()
    return got


def test_a_call_under_its_needed_size(cg):
    u = field(1)
    plain = needed(cg)
    mesh = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    full, rep_full = smooth(cg, mesh, u)
    mesh.close()
    cg.set_workspace_limit(cg.workspace_bytes() + plain)
    mesh = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    for _ in range(3):
        tight, rep = smooth(cg, mesh, u)
        assert near(tight, full, u)
        assert rep["iters"] > rep_full["iters"]        # own first rounds
    cg.set_workspace_limit(0)                          # the refusal is forgotten
    again, rep = smooth(cg, mesh, u)
    assert rep["iters"] == rep_full["iters"]
    assert bool((again == full).all())
    mesh.close()


def test_another_mesh_takes_optional_memory_back(cg):
    u = field(2)
    plain = needed(cg)
    held = cg.workspace_bytes()
    a = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    full, rep_full = smooth(cg, a, u)
    assert cg.workspace_bytes() - held > 2 * plain     # the expansion's vectors are the larger part
    cg.set_workspace_limit(held + 2 * plain)
    b = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    for mesh in (b, a, b):
        x, rep = smooth(cg, mesh, u)
        assert near(x, full, u)
        assert cg.workspace_bytes() <= held + 2 * plain
    x = u.clone()
    c = cg.StructuredMesh((8, 8, 8), (0, 0, 0), 1.0)
    with pytest.raises(cg.CGError) as e:               # nothing optional is left to take back
        cg.diffuse(c, x[:, :512].clone(), cg.Params(T=2.0, nsteps=NSTEPS, precision=3))
    assert e.value.code == "CG_ENOMEM"
    cg.set_workspace_limit(0)
    x, rep = smooth(cg, a, u)
    assert bool((x == full).all()) and rep["iters"] == rep_full["iters"]
    for m in (a, b, c):
        m.close()
    assert cg.workspace_bytes() == held


def test_concurrent_calls_wait_for_optional_memory_in_use(cg):
    """Several problems at a time under a limit that holds the needed vectors of all."""
    import torch
    k = 4
    rng = np.random.default_rng(3)
    pos = torch.from_numpy(rng.random((3, 50_000)) * np.array(DIMS)[:, None]).cuda()
    w = torch.from_numpy(rng.random((1, 50_000))).cuda()
    par = [cg.Params(T=t, nsteps=NSTEPS, precision=3) for t in (1.0, 2.0, 3.0, 4.0)]
    cap = [cg.Params(T=t, nsteps=NSTEPS, precision=3, max_iter=CAP) for t in (1.0, 2.0, 3.0, 4.0)]
    streams = [torch.cuda.Stream() for _ in range(k)]
    held = cg.workspace_bytes()

    def run(p):
        meshes = [cg.StructuredMesh(DIMS, (0, 0, 0), 1.0) for _ in range(k)]
        out = cg.coarse_grain_concurrent(meshes, [pos] * k, [w] * k, p, streams=streams, max_concurrent=k)
        size = cg.workspace_bytes() - held
        for m in meshes:
            m.close()
        return out, size

    ref, size = run(cap)
    cg.set_workspace_limit(held + size)
    got, _ = run(par)
    for a, b in zip(got, ref):
        assert near(a, b, b)


def test_fp64_beyond_the_cooperative_size(cg):
    import torch
    dims = (104, 96, 100)
    n = dims[0] * dims[1] * dims[2]
    u = torch.from_numpy(np.random.default_rng(4).random((1, n))).cuda()
    a = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    held = cg.workspace_bytes()
    smooth(cg, a, field(5))
    taken = cg.workspace_bytes() - held
    a.close()
    cg.set_workspace_limit(held + taken)
    a = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    smooth(cg, a, field(5))
    assert cg.workspace_bytes() == held + taken
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)     # three vectors fit once the expansion's are back
    x = u.clone()
    cg.diffuse(mesh, x, cg.Params(T=2.0, nsteps=NSTEPS))
    cg.set_workspace_limit(0)
    y = u.clone()
    cg.diffuse(mesh, y, cg.Params(T=2.0, nsteps=NSTEPS))
    assert near(x, y, u)
    mesh.close()
    a.close()


def test_a_limit_of_what_is_held_and_some_more(cg):
    """Optional memory held when the limit is set counts as held: room for x is room for x."""
    import torch
    a = cg.StructuredMesh(DIMS, (0, 0, 0), 1.0)
    smooth(cg, a, field(7))
    held = cg.workspace_bytes()
    b = cg.StructuredMesh((32, 32, 32), (0, 0, 0), 1.0)
    u = torch.zeros((1, 32 ** 3), dtype=torch.float64, device="cuda")
    cg.set_workspace_limit(held + 64 * 1024)
    with pytest.raises(cg.CGError) as e:
        cg.diffuse(b, u, cg.Params(T=2.0, nsteps=NSTEPS, precision=3))
    assert e.value.code == "CG_ENOMEM"
    assert held <= cg.workspace_bytes() <= held + 64 * 1024
    a.close()
    b.close()


def test_a_batch_under_its_needed_size(cg):
    """Snapshots of which the first is the largest; one round a step, which no step ends
    with, never takes the expansion: its workspace is what the batch needs."""
    import torch
    rng = np.random.default_rng(6)
    dims = [(80, 72, 64), (40, 30, 33), (64, 64, 60), (20, 21, 22), (90, 50, 40)]
    us = [torch.from_numpy(rng.random((2, a * b * c))).cuda() for a, b, c in dims]
    held = cg.workspace_bytes()

    def run(meshes, **kw):
        x = [u.clone() for u in us]
        _, rep = cg.diffuse_batched(meshes, x, cg.Params(nsteps=6, precision=3, sweep_shape=508, **kw),
                                    bandwidths=[2.5] * len(dims), report=True)
        return x, rep

    def meshes_of():
        return [cg.StructuredMesh(d, (0, 0, 0), 1.0) for d in dims]

    meshes = meshes_of()
    with pytest.raises(cg.CGError):
        run(meshes, max_rounds=1)
    plain = cg.workspace_bytes() - held
    full, rep_full = run(meshes)
    extra = cg.workspace_bytes() - held - plain
    for m in meshes:
        m.close()
    assert extra > 0
    for room in (0, extra // 3):              # none for the expansion; some, not enough
        cg.set_workspace_limit(held + plain + room)
        meshes = meshes_of()
        sizes = []
        for _ in range(3):
            got, rep = run(meshes)
            sizes.append(cg.workspace_bytes() - held)
            assert rep["iters"] > rep_full["iters"]
            for a, b, u in zip(got, full, us):
                assert near(a, b, u)
        assert sizes[0] == sizes[1] == sizes[2] <= plain + room
        cg.set_workspace_limit(0)
        got, rep = run(meshes)
        assert rep["iters"] == rep_full["iters"]
        assert all(bool((a == b).all()) for a, b in zip(got, full))
        for m in meshes:
            m.close()
    assert cg.workspace_bytes() == held
