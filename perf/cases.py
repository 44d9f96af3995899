"""Performance cases: coarse-graining work as a user's program calls it, through the
package's public entry points, with its inputs, its minimal work and its exact results.

The sizes and distributions are those of the workloads of this repository (``workloads/``)
or lie between them: particles in a cube or a channel, one to five carried fields,
uniform, periodic, stretched and tetrahedral meshes, single calls, concurrent calls and
batches.  ``exact`` restates the method in 64 bits with torch and numpy alone: particle
centroid deposition, then the implicit Euler, Crank-Nicolson or explicit Euler steps, by
the eigenvectors of the per-axis second difference on uniform meshes and by conjugate
gradients on the others.
"""
import math

import numpy as np
import torch

import paper_1409_0001_gb300 as cg

IE, CN, EXPLICIT = cg.SCHEME_IMPLICIT_EULER, cg.SCHEME_CRANK_NICOLSON, cg.SCHEME_EXPLICIT_EULER
FP64, FP32_REFINE, FP32_DF, BF16_DF = (cg.PREC_FP64, cg.PREC_FP32_REFINE, cg.PREC_FP32_DF_REFINE,
                                       cg.PREC_BF16_DF_REFINE)
ORDERED, FIXED = cg.DEPOSIT_ORDERED, cg.DEPOSIT_FIXED_POINT


def _grain(name, dims, n, b, nsteps, fields=1, precision=FP32_DF, scheme=IE, deposit=ORDERED,
           fused_k=0, particles="uniform", period="", host=False, velocity=False):
    """One call on a uniform mesh: dims cells of edge 1 / max(dims) (the channel's box is
    twice as long as high), b in cells."""
    return {"name": name, "kind": "grain", "nx": dims[0], "ny": dims[1], "nz": dims[2], "n": n,
            "b": b, "nsteps": nsteps, "fields": fields, "precision": precision, "scheme": scheme,
            "deposit": deposit, "fused_k": fused_k, "particles": particles, "period": period,
            "host": host, "velocity": velocity}


def listed():
    return [
        # the smallest call: the particles of a small solver step onto a coarse mesh, no
        # smoothing (launches, synchronisations and host work count here)
        {"name": "deposit_32", "kind": "deposit", "nx": 32, "ny": 32, "nz": 32, "n": 10_000,
         "fields": 1, "deposit": ORDERED},
        # the plain FP64 method at the smallest stated size, with the default parameters
        _grain("cube32_fp64", (32, 32, 32), 10_000, 3.0, 10, precision=FP64),
        # a mid-size mesh with odd, unequal sides (no vector width divides a row), the
        # scheme the paper itself uses, volume and two momentum components
        _grain("ragged_cn", (97, 61, 45), 150_000, 3.0, 10, fields=3, scheme=CN),
        # one bandwidth of the clustered cube from pinned host arrays and back: a solver
        # whose particles live on the host
        _grain("cube128_host", (128, 128, 128), 2_000_000, 2.0, 10, particles="clustered", host=True),
        # the benchmark step: four bandwidths of the clustered cube, two at a time
        {"name": "cube128_step", "kind": "concurrent", "side": 128, "n": 2_000_000, "nsteps": 10,
         "b0": 1.0, "nb": 4, "workers": 2},
        # the plain FP64 method where arithmetic and memory count instead of launches
        _grain("cube96_fp64", (96, 96, 96), 1_000_000, 4.0, 10, precision=FP64),
        # a channel periodic along the flow: volume and momentum, then the solid velocity
        _grain("channel_periodic", (256, 128, 128), 6_000_000, 4.0, 20, fields=4,
               particles="channel", period="x", velocity=True),
        # reduced storage of the inner vectors, as the large-channel workload states it
        _grain("channel256_bf16", (256, 128, 128), 6_000_000, 4.0, 20, precision=BF16_DF,
               particles="channel"),
        # explicit steps (blocked, FP32) after an exact integer deposition of five fields
        _grain("explicit_fixed", (256, 128, 128), 4_000_000, 4.0, 40, fields=2, scheme=EXPLICIT,
               deposit=FIXED, fused_k=3, particles="channel"),
        # an unstructured mesh with a dense bottom layer
        {"name": "tet", "kind": "tet", "side": 48, "n": 600_000, "b": 3.0, "nsteps": 10, "fields": 1},
        # a batch of independent snapshots of uneven size with five fields each
        {"name": "batch64", "kind": "batch", "snaps": 64, "side_lo": 32, "side_hi": 96,
         "logn_lo": 4.0, "logn_hi": 6.0, "b": 3.0, "nsteps": 10, "fields": 5},
        # the large channel: fifty million particles, forty steps
        _grain("channel512", (512, 256, 256), 50_000_000, 4.0, 40, particles="channel"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["deposit", "grain", "grain", "grain", "grain_fp64", "periodic", "bf16",
                       "explicit", "concurrent", "tet", "hex", "batch"])
    nsteps = rng.choice([5, 8, 10, 12, 16, 20])
    # b at most 4 nsteps^(1/2) / 2.2 cells: dtau / dx^2 at most about 0.8
    b = round(rng.uniform(1.0, min(6.0, 1.8 * math.sqrt(nsteps))), 2)
    dims = [_logint(rng, 24, 192) for _ in range(3)]
    if rng.random() < 0.5:   # rows that a vector width divides, half of the time
        dims[0] = max(4, dims[0] // 4 * 4)
    cells = dims[0] * dims[1] * dims[2]
    n = min(20_000_000, max(5_000, int(cells * math.exp(rng.uniform(math.log(0.2), math.log(3.0))))))
    fields = rng.choice([1, 1, 1, 3, 4, 5])
    if kind == "deposit":
        return {"kind": "deposit", "nx": dims[0], "ny": dims[1], "nz": dims[2], "n": n,
                "fields": fields, "deposit": rng.choice([ORDERED, FIXED])}
    if kind == "concurrent":
        return {"kind": "concurrent", "side": rng.choice([64, 80, 96, 100, 128]),
                "n": _logint(rng, 50_000, 2_000_000), "nsteps": 10,
                "b0": round(rng.uniform(0.5, 1.0), 2), "nb": rng.choice([2, 3, 4]), "workers": 2}
    if kind == "tet":
        return {"kind": "tet", "side": rng.randint(8, 48), "n": _logint(rng, 10_000, 600_000),
                "b": round(rng.uniform(2.0, 4.0), 2), "nsteps": rng.choice([5, 10]),
                "fields": rng.choice([1, 1, 3])}
    if kind == "hex":
        return {"kind": "hex", "side": rng.randint(20, 80), "n": _logint(rng, 20_000, 800_000),
                "b": round(rng.uniform(1.5, 2.5), 2), "nsteps": 10, "fields": rng.choice([1, 4]),
                "ratio": round(rng.uniform(1.0, 1.04), 3)}
    if kind == "batch":
        lo = rng.randint(16, 48)
        return {"kind": "batch", "snaps": rng.randint(4, 40), "side_lo": lo,
                "side_hi": lo + rng.randint(4, 32), "logn_lo": 3.5, "logn_hi": 5.5,
                "b": round(rng.uniform(1.5, 4.0), 2), "nsteps": rng.choice([5, 10]),
                "fields": rng.choice([1, 4, 5])}
    if kind == "explicit":
        steps = rng.choice([20, 30, 40])
        case = _grain("", dims, n, round(rng.uniform(1.5, 1.6 * math.sqrt(steps) / 2), 2), steps,
                      fields=min(fields, 3), scheme=EXPLICIT, deposit=rng.choice([ORDERED, FIXED]),
                      precision=FP32_DF, fused_k=rng.choice([0, 1, 3, 4]))
    elif kind == "periodic":
        case = _grain("", dims, max(n, cells), max(b, 3.0), max(nsteps, 10), fields=4,
                      period=rng.choice(["x", "x", "xy", "xyz"]), particles="channel", velocity=True)
    elif kind == "bf16":
        case = _grain("", dims, n, b, nsteps, fields=min(fields, 3), precision=BF16_DF)
    elif kind == "grain_fp64":
        dims = [min(d, 96) for d in dims]
        case = _grain("", dims, min(n, 1_000_000), b, nsteps, fields=min(fields, 3), precision=FP64,
                      scheme=rng.choice([IE, IE, CN]))
    else:
        case = _grain("", dims, n, b, nsteps, fields=fields, scheme=rng.choice([IE, IE, CN]),
                      deposit=rng.choice([ORDERED, ORDERED, FIXED]),
                      particles=rng.choice(["uniform", "clustered"]), host=rng.random() < 0.2)
    del case["name"]
    return case


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 1)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


def _randn(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _box(case):
    """Cell edge and box lengths; edges are powers of two where the sides allow it."""
    d = max(case["nx"], case["ny"], case["nz"])
    dx = (4.0 if case.get("particles") == "channel" else 1.0) / d
    return dx, [case["nx"] * dx, case["ny"] * dx, case["nz"] * dx]


def _inside(pos, lengths):
    for a in range(3):   # the boxes start at 0; a centroid on or past the far wall moves in
        pos[a].clamp_(0.0, lengths[a] * (1 - 1e-12))
    return pos


def _uniform(g, n, lengths):
    pos = _rand(g, 3, n)
    for a in range(3):
        pos[a] *= lengths[a]
    return _inside(pos, lengths)


def _channel(g, n, lengths):
    """Density proportional to 1 + 0.5 sin(2 pi x) along the channel."""
    pos = _uniform(g, n, lengths)
    got, xs = 0, []
    while got < n:
        x = _rand(g, 2 * (n - got) + 1024) * lengths[0]
        x = x[_rand(g, x.numel()) * 1.5 < 1.0 + 0.5 * torch.sin(2 * math.pi * x)][:n - got]
        xs.append(x)
        got += x.numel()
    pos[0] = torch.cat(xs)
    return _inside(pos, lengths)


def _clustered(g, n, lengths, dims, cap):
    """20 Gaussian clusters (sigma 0.05 of a side), at most `cap` centroids in a cell; what
    falls outside or into a full cell is drawn again, in the end uniformly."""
    L = torch.tensor(lengths, dtype=torch.float64, device="cuda")[:, None]
    dim = torch.tensor(dims, device="cuda")[:, None]
    centre = 0.1 + 0.8 * _rand(g, 3, 20)
    which = torch.randint(0, 20, (n,), device="cuda", generator=g)
    pos = torch.empty(3, n, dtype=torch.float64, device="cuda")
    todo = torch.arange(n, device="cuda")
    full = torch.zeros(dims[0] * dims[1] * dims[2], dtype=torch.int64, device="cuda")
    for attempt in range(10):
        m = todo.numel()
        if m == 0:
            break
        p = centre[:, which[todo]] + 0.05 * _randn(g, 3, m) if attempt < 6 else _rand(g, 3, m)
        ok = ((p >= 0) & (p < 1)).all(0)
        ijk = (p.clamp(0, 1 - 1e-9) * dim).long()
        cell = (ijk[2] * dims[1] + ijk[1]) * dims[0] + ijk[0]
        order = torch.argsort(cell, stable=True)
        s = cell[order]
        rank = torch.empty_like(s)
        rank[order] = torch.arange(m, device="cuda") - torch.searchsorted(s, s)
        ok &= (full[cell] + rank < cap) | (attempt == 9)
        pos[:, todo] = p
        full.index_add_(0, cell[ok], torch.ones_like(cell[ok]))
        todo = todo[~ok]
    return _inside(pos * L, lengths)


def _weights(g, n, fields, d, pos=None):
    """V_p, V_p u (u ~ N(0, 0.1), streamwise 1 + 0.5 sin(2 pi x) in a channel), drag."""
    vp = math.pi * d ** 3 / 6.0
    w = torch.full((fields, n), vp, dtype=torch.float64, device="cuda")
    for f in range(1, min(fields, 4)):
        u = 0.1 * _randn(g, n)
        if f == 1 and pos is not None:
            u += 1.0 + 0.5 * torch.sin(2 * math.pi * pos[0])
        w[f] *= u
    if fields == 5:
        w[4] = torch.exp(_randn(g, n))
    return w


def _particles(case, seed):
    g = _gen(seed)
    dx, lengths = _box(case)
    dims, n = (case["nx"], case["ny"], case["nz"]), case["n"]
    how = case.get("particles", "uniform")
    if how == "channel":
        pos = _channel(g, n, lengths)
    elif how == "clustered":
        pos = _clustered(g, n, lengths, dims, max(8, 4 * n // (dims[0] * dims[1] * dims[2])))
    else:
        pos = _uniform(g, n, lengths)
    w = _weights(g, n, case["fields"], 0.3 * dx, pos if how == "channel" else None)
    return pos.contiguous(), w


def _period(case):
    return tuple(a in case.get("period", "") for a in "xyz")


def _layered(g, n, fields):
    """70 % of the particles in the bottom fifth of the unit cube."""
    pos = _uniform(g, n, [1.0, 1.0, 1.0])
    pos[2, : int(0.7 * n)] *= 0.2
    return pos, _weights(g, n, fields, 0.003)


def _tet_mesh(side, seed):
    """The unit cube's side^3 hexes, six tetrahedra each (one per axis permutation),
    interior vertices moved by up to 0.15 of a hex edge."""
    rng = np.random.default_rng(seed)
    t = np.arange(side + 1)
    k, j, i = np.meshgrid(t, t, t, indexing="ij")
    ijk = np.stack([i, j, k], -1).reshape(-1, 3)
    xyz = ijk / side
    inner = np.all((ijk > 0) & (ijk < side), axis=1)
    xyz[inner] += rng.uniform(-0.15, 0.15, (int(inner.sum()), 3)) / side
    h = np.arange(side)
    k, j, i = np.meshgrid(h, h, h, indexing="ij")
    base = ((k * (side + 1) + j) * (side + 1) + i).ravel()
    step = (1, side + 1, (side + 1) ** 2)
    tets = np.empty((base.size, 6, 4), dtype=np.int32)
    for p, (a, b, c) in enumerate([(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]):
        tets[:, p, 0] = base
        tets[:, p, 1] = base + step[a]
        tets[:, p, 2] = base + step[a] + step[b]
        tets[:, p, 3] = base + step[a] + step[b] + step[c]
    return xyz, tets.reshape(-1, 4)


def _hex_faces(case):
    """Uniform faces in x and y, z faces growing away from the bottom wall; D = 1 with a
    block of 0 and a slab of 4."""
    n = case["side"]
    x = np.linspace(0.0, 1.0, n + 1)
    z = np.concatenate([[0.0], np.cumsum(case["ratio"] ** np.arange(n))])
    z /= z[-1]
    z[-1] = 1.0
    D = np.ones((n, n, n))
    D[n // 8:n // 4, 3 * n // 8:5 * n // 8, 3 * n // 8:5 * n // 8] = 0.0
    D[n // 2:3 * n // 4, n // 8:n // 4, :] = 4.0
    return x, z, D


def _sizes(case):
    """The batch's (side, particles) per snapshot: the same for every seed."""
    rng = np.random.default_rng(case["snaps"])
    return [(int(rng.integers(case["side_lo"], case["side_hi"] + 1)),
             int(round(10.0 ** rng.uniform(case["logn_lo"], case["logn_hi"]))))
            for _ in range(case["snaps"])]


def _snapshots(case, seed):
    got = []
    for s, (side, n) in enumerate(_sizes(case)):
        g = _gen(seed * 1009 + s)
        pos = _uniform(g, n, [1.0, 1.0, 1.0])
        got.append((side, pos, _weights(g, n, case["fields"], 0.004)))
    return got


# ------------------------------------------------------------------------------ the path
def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind in ("grain", "deposit"):
        pos, w = _particles(case, seed)
        dx, _ = _box(case)
        st["mesh"] = cg.StructuredMesh((case["nx"], case["ny"], case["nz"]), (0.0, 0.0, 0.0), dx,
                                       periodic=_period(case))
        if case.get("host"):
            pos, w = pos.cpu().pin_memory(), w.cpu().pin_memory()
            st["out"] = torch.empty((case["fields"], st["mesh"].ncells), dtype=torch.float64,
                                    pin_memory=True)
        st["pos"], st["w"] = pos, w
        if kind == "deposit":
            st["params"] = cg.Params(deposit_mode=case["deposit"])
        else:
            st["params"] = cg.Params(bandwidth=case["b"] * dx, nsteps=case["nsteps"],
                                     scheme=case["scheme"], precision=case["precision"],
                                     deposit_mode=case["deposit"], fused_k=case["fused_k"])
            st["host"], st["velocity"] = case["host"], case["velocity"]
    elif kind == "concurrent":
        n_side = case["side"]
        dims = (n_side,) * 3
        g = _gen(seed)
        st["pos"] = _clustered(g, case["n"], [1.0] * 3, dims, max(8, 4 * case["n"] // n_side ** 3))
        st["w"] = _weights(g, case["n"], 1, 0.004)
        st["meshes"] = [cg.StructuredMesh(dims, (0.0,) * 3, 1.0 / n_side) for _ in range(case["nb"])]
        st["streams"] = [torch.cuda.Stream() for _ in range(case["nb"])]
        st["params"] = [cg.Params(bandwidth=b / n_side, nsteps=case["nsteps"], precision=FP32_DF)
                        for b in _bandwidths(case)]
        st["workers"] = case["workers"]
    elif kind == "tet":
        st["pos"], st["w"] = _layered(_gen(seed), case["n"], case["fields"])
        st["mesh"] = cg.TetMesh(*_tet_mesh(case["side"], seed))
        st["params"] = cg.Params(bandwidth=case["b"] / case["side"], nsteps=case["nsteps"],
                                 precision=FP32_REFINE)
    elif kind == "hex":
        st["pos"], st["w"] = _layered(_gen(seed), case["n"], case["fields"])
        x, z, D = _hex_faces(case)
        st["mesh"] = cg.HexMesh(x, x, z, D.ravel())
        st["params"] = cg.Params(bandwidth=case["b"] / case["side"], nsteps=case["nsteps"],
                                 precision=FP32_REFINE)
    else:
        snaps = _snapshots(case, seed)
        st["meshes"] = [cg.StructuredMesh((s,) * 3, (0.0,) * 3, 1.0 / s) for s, _, _ in snaps]
        st["pos"], st["w"] = [p for _, p, _ in snaps], [w for _, _, w in snaps]
        st["bandwidths"] = [case["b"] / s for s, _, _ in snaps]
        st["params"] = cg.Params(nsteps=case["nsteps"], precision=FP32_DF)
    torch.cuda.synchronize()
    return st


def _bandwidths(case):
    return [case["b0"] * 2.0 ** q for q in range(case["nb"])]


def run(st):
    kind = st["kind"]
    if kind == "deposit":
        return cg.deposit(st["mesh"], st["pos"], st["w"], st["params"])
    if kind == "concurrent":
        k = len(st["meshes"])
        return cg.coarse_grain_concurrent(st["meshes"], [st["pos"]] * k, [st["w"]] * k, st["params"],
                                          streams=st["streams"], max_concurrent=st["workers"])
    if kind == "batch":
        return cg.coarse_grain_batched(st["meshes"], st["pos"], st["w"], st["params"],
                                       bandwidths=st["bandwidths"])
    if kind == "grain" and st["host"]:
        return cg.coarse_grain_host(st["mesh"], st["pos"], st["w"], st["params"], out=st["out"])
    cells = cg.coarse_grain(st["mesh"], st["pos"], st["w"], st["params"])
    if kind == "grain" and st["velocity"]:
        return {"cells": cells, "velocity": cg.solid_velocity(st["mesh"], cells[0], cells[1:])}
    return cells


def work(case):
    """Each particle's position and weights read once, each cell value written once (a
    mesh given by its vertices or faces read once); one operator application per step."""
    kind, F = case["kind"], case.get("fields", 1)
    extra, steps = 0.0, case.get("nsteps", 0)
    outs = F
    if kind == "concurrent":
        cells, n, outs = case["side"] ** 3, case["n"], case["nb"]
    elif kind == "batch":
        cells, n = sum(s ** 3 for s, _ in _sizes(case)), sum(p for _, p in _sizes(case))
    elif kind == "tet":
        cells, n = 6 * case["side"] ** 3, case["n"]
        extra = 16.0 * cells + 24.0 * (case["side"] + 1) ** 3
    elif kind == "hex":
        cells, n = case["side"] ** 3, case["n"]
        extra = 8.0 * cells
    else:
        cells, n = case["nx"] * case["ny"] * case["nz"], case["n"]
        if case.get("velocity"):
            extra = 8.0 * (F - 1) * cells
    return {"bytes": (24.0 + 8.0 * F) * n + 8.0 * outs * cells + extra,
            "flops": 1.0 * F * n + (1.0 + 9.0 * steps) * outs * cells}


# ------------------------------------------------------------------------------ 64 bits
def _sum_cells(cell, w, ncells, volume):
    out = torch.zeros(w.shape[0], ncells, dtype=torch.float64, device="cuda")
    for f in range(w.shape[0]):
        out[f].index_add_(0, cell, w[f])
    return out / volume


def _deposit_uniform(pos, w, dims, dx):
    ijk = [(pos[a] * (1.0 / dx)).floor().long().clamp_(0, dims[a] - 1) for a in range(3)]
    cell = (ijk[2] * dims[1] + ijk[1]) * dims[0] + ijk[0]
    return _sum_cells(cell, w, dims[0] * dims[1] * dims[2], (dx * dx) * dx)


def _axis(n, periodic):
    """Orthonormal eigenvectors (columns) and eigenvalues of the negative second
    difference: cosines between walls, cos + sin on a periodic axis."""
    j = torch.arange(n, dtype=torch.float64, device="cuda")
    if periodic:
        ang = 2 * math.pi * (j[:, None] * j[None, :] % n) / n
        return (torch.cos(ang) + torch.sin(ang)) / math.sqrt(n), 4 * torch.sin(math.pi * j / n) ** 2
    q = torch.cos(math.pi * (j[:, None] + 0.5) * j[None, :] / n) * math.sqrt(2.0 / n)
    q[:, 0] = math.sqrt(1.0 / n)
    return q, 4 * torch.sin(math.pi * j / (2 * n)) ** 2


def _smooth_uniform(cells, dims, periodic, b, nsteps, scheme):
    """nsteps steps to T = b^2 / 4 (b in cells) by the separable eigenvectors."""
    c = b * b / 4.0 / nsteps
    (qx, lx), (qy, ly), (qz, lz) = [_axis(dims[a], periodic[a]) for a in range(3)]
    mu = c * (lz[:, None, None] + ly[None, :, None] + lx[None, None, :])
    gain = (1 / (1 + mu) if scheme == IE else (1 - mu / 2) / (1 + mu / 2) if scheme == CN else 1 - mu) ** nsteps
    out = torch.empty_like(cells)
    for f in range(cells.shape[0]):
        u = cells[f].view(dims[2], dims[1], dims[0])
        u = torch.matmul(u, qx)
        u = torch.matmul(qy.T, u)
        u = torch.matmul(qz.T, u.reshape(dims[2], -1)).view(dims[2], dims[1], dims[0])
        u = u * gain
        u = torch.matmul(qz, u.reshape(dims[2], -1)).view(dims[2], dims[1], dims[0])
        u = torch.matmul(qy, u)
        out[f] = torch.matmul(u, qx.T).reshape(-1)
    return out


def _implicit(cells, volume, dtau, nsteps, apply_l, diag):
    """Implicit Euler (M - dtau L) u = M u_n, field by field, by Jacobi-preconditioned
    conjugate gradients to the end of 64 bits."""
    inv = 1.0 / (volume + dtau * diag)
    out = torch.empty_like(cells)
    for f in range(cells.shape[0]):
        u = cells[f].clone()
        for _ in range(nsteps):
            rhs = volume * u
            r = rhs - (volume * u - dtau * apply_l(u))
            z = inv * r
            p = z.clone()
            rz = torch.dot(r, z)
            stop = 1e-31 * torch.dot(rhs, inv * rhs).item()
            for it in range(400):
                if it % 8 == 0 and rz.item() <= stop:
                    break
                q = volume * p - dtau * apply_l(p)
                alpha = rz / torch.dot(p, q)
                u = u + alpha * p
                r = r - alpha * q
                z = inv * r
                new = torch.dot(r, z)
                p = z + (new / rz) * p
                rz = new
        out[f] = u
    return out


def _exact_hex(case, pos, w):
    n = case["side"]
    x, z, D = _hex_faces(case)
    faces = [torch.from_numpy(v).cuda() for v in (x, x, z)]
    ijk = [(torch.searchsorted(faces[a], pos[a].contiguous(), right=True) - 1).clamp_(0, n - 1)
           for a in range(3)]
    h = [v[1:] - v[:-1] for v in faces]
    volume = (h[2][:, None, None] * h[1][None, :, None] * h[0][None, None, :]).reshape(-1)
    cells = _sum_cells((ijk[2] * n + ijk[1]) * n + ijk[0], w, n ** 3, volume)
    d = torch.from_numpy(D).cuda()
    T = []
    for a, axis in ((0, 2), (1, 1), (2, 0)):   # transmissibilities across each axis' inner faces
        lo, hi = d.narrow(axis, 0, n - 1), d.narrow(axis, 1, n - 1)
        harm = torch.where((lo > 0) & (hi > 0), 2 * lo * hi / (lo + hi).clamp_min(1e-300), torch.zeros_like(lo))
        dist = 0.5 * (h[a][1:] + h[a][:-1])
        shape = [1, 1, 1]
        shape[axis] = n - 1
        area = torch.ones(n, n, n, dtype=torch.float64, device="cuda")
        for o, oaxis in ((0, 2), (1, 1), (2, 0)):
            if o != a:
                s = [1, 1, 1]
                s[oaxis] = n
                area = area * h[o].view(s)
        T.append((axis, harm * area.narrow(axis, 0, n - 1) / dist.view(shape)))

    def flux(u):
        u = u.view(n, n, n)
        out = torch.zeros_like(u)
        for axis, t in T:
            fl = t * (u.narrow(axis, 1, n - 1) - u.narrow(axis, 0, n - 1))
            out.narrow(axis, 0, n - 1).add_(fl)
            out.narrow(axis, 1, n - 1).sub_(fl)
        return out.reshape(-1)

    diag = torch.zeros(n, n, n, dtype=torch.float64, device="cuda")
    for axis, t in T:
        diag.narrow(axis, 0, n - 1).add_(t)
        diag.narrow(axis, 1, n - 1).add_(t)
    b = case["b"] / n
    return _implicit(cells, volume, b * b / 4 / case["nsteps"], case["nsteps"], flux, diag.reshape(-1))


def _exact_tet(case, seed, pos, w):
    n = case["side"]
    xyz, tets = _tet_mesh(n, seed)
    X = torch.from_numpy(xyz).cuda()
    V = torch.from_numpy(tets.astype(np.int64)).cuda()
    corner = X[V]                                        # [tets, 4, 3]
    edges = corner[:, 1:] - corner[:, :1]
    volume = torch.linalg.det(edges).abs() / 6.0
    inv = torch.linalg.inv(edges)                        # barycentric: (x - x0) @ inv
    # host tet: the tets of the 27 hexes around the point, largest least coordinate
    m = pos.shape[1]
    cell = torch.empty(m, dtype=torch.int64, device="cuda")
    for s in range(0, m, 50_000):
        p = pos[:, s:s + 50_000].T
        home = (p * n).long().clamp_(0, n - 1)
        best = torch.full((p.shape[0],), -math.inf, dtype=torch.float64, device="cuda")
        who = torch.zeros(p.shape[0], dtype=torch.int64, device="cuda")
        for off in range(27):
            q = home + torch.tensor([off % 3 - 1, off // 3 % 3 - 1, off // 9 - 1], device="cuda")
            ok = ((q >= 0) & (q < n)).all(1)
            q = q.clamp(0, n - 1)
            first = ((q[:, 2] * n + q[:, 1]) * n + q[:, 0]) * 6
            for t in range(6):
                lam = torch.matmul((p - corner[first + t, 0])[:, None, :], inv[first + t])[:, 0]
                low = torch.minimum(lam.min(1).values, 1 - lam.sum(1))
                low = torch.where(ok, low, torch.full_like(low, -math.inf))
                better = low > best
                best = torch.where(better, low, best)
                who = torch.where(better, first + t, who)
        cell[s:s + 50_000] = who
    cells = _sum_cells(cell, w, V.shape[0], volume)
    # two-point fluxes between the tets that share a face
    nt = V.shape[0]
    opposite = [[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]]
    tri = torch.cat([V[:, o] for o in opposite]).sort(1).values
    key = (tri[:, 0] * X.shape[0] + tri[:, 1]) * X.shape[0] + tri[:, 2]
    key, order = key.sort()
    pair = (key[1:] == key[:-1]).nonzero()[:, 0]
    fa, fb = order[pair], order[pair + 1]
    ca, cb = fa % nt, fb % nt
    f = X[tri[fa]]
    area = 0.5 * torch.linalg.cross(f[:, 1] - f[:, 0], f[:, 2] - f[:, 0])
    mid = corner.mean(1)
    d = mid[cb] - mid[ca]
    T = (area * area).sum(1) / (area * d).sum(1).abs()
    diag = torch.zeros(nt, dtype=torch.float64, device="cuda").index_add_(0, ca, T).index_add_(0, cb, T)
    L = torch.sparse_coo_tensor(torch.stack([torch.cat([ca, cb]), torch.cat([cb, ca])]),
                                torch.cat([T, T]), (nt, nt)).coalesce().to_sparse_csr()
    b = case["b"] / n
    return _implicit(cells, volume, b * b / 4 / case["nsteps"], case["nsteps"],
                     lambda u: torch.mv(L, u) - diag * u, diag)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("grain", "deposit"):
        pos, w = _particles(case, seed)
        dx, _ = _box(case)
        dims = (case["nx"], case["ny"], case["nz"])
        cells = _deposit_uniform(pos, w, dims, dx)
        if kind == "deposit":
            return cells
        cells = _smooth_uniform(cells, dims, _period(case), case["b"], case["nsteps"], case["scheme"])
        if case["velocity"]:
            return {"cells": cells, "velocity": cells[1:] / cells[0]}
        return cells.cpu() if case["host"] else cells
    if kind == "concurrent":
        n = case["side"]
        g = _gen(seed)
        pos = _clustered(g, case["n"], [1.0] * 3, (n,) * 3, max(8, 4 * case["n"] // n ** 3))
        cells = _deposit_uniform(pos, _weights(g, case["n"], 1, 0.004), (n,) * 3, 1.0 / n)
        return [_smooth_uniform(cells, (n,) * 3, (False,) * 3, b, case["nsteps"], IE)
                for b in _bandwidths(case)]
    if kind == "batch":
        return [_smooth_uniform(_deposit_uniform(pos, w, (s,) * 3, 1.0 / s), (s,) * 3, (False,) * 3,
                                case["b"], case["nsteps"], IE)
                for s, pos, w in _snapshots(case, seed)]
    pos, w = _layered(_gen(seed), case["n"], case["fields"])
    return _exact_hex(case, pos, w) if kind == "hex" else _exact_tet(case, seed, pos, w)
