"""GPU: the conversions between FP64 and double-float, bit for bit against their FP64
definition (hi = fl32(v), lo = fl32(v - hi), back fl64(hi + lo)): a constant field on cells of
at most one neighbour (no sum rounds) is left as it is by a smoothing, so a call returns
exactly its converted value.  Values across the
integer path's exponents and beyond both ends, ties of the significand's rounding, powers
of two and their neighbours, zeros.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def values():
    rng = np.random.default_rng(11)
    v = [np.ldexp(1.0 + rng.random(200), rng.integers(-69, 126, 200)) * rng.choice([-1, 1], 200),
         np.ldexp(1.0 + rng.random(40), rng.integers(-100, -70, 40)),
         np.ldexp(1.0, np.arange(-74, 120, 5)), -np.ldexp(1.0, np.arange(-60, 60, 7))]
    base = 1.0 + rng.integers(0, 1 << 23, 64) * 2.0 ** -23      # ties of the 24-bit rounding
    for off in (2.0 ** -24, 2.0 ** -24 + 2.0 ** -52, 2.0 ** -24 - 2.0 ** -52, -2.0 ** -53):
        v += [base + off, -(base + off)]
    v += [np.array([0.0, -0.0, 1.0, np.nextafter(1.0, 0), np.nextafter(2.0, 0), np.nextafter(2.0 ** 24, 0)])]
    return np.concatenate(v)


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 1, 1), (1, 2, 1)])
def test_round_trip(dims):
    import torch

    import paper_1409_0001_gb300 as cg
    v = values()
    hi = v.astype(np.float32)
    lo = (v - hi.astype(np.float64)).astype(np.float32)
    ref = hi.astype(np.float64) + lo.astype(np.float64)
    n = dims[0] * dims[1] * dims[2]
    mesh = cg.StructuredMesh(dims, (0, 0, 0), 1.0)
    for i in range(0, len(v), 64):
        u = np.repeat(v[i:i + 64, None], n, axis=1)
        x = torch.from_numpy(u).cuda()
        cg.diffuse(mesh, x, cg.Params(T=0.5, nsteps=2, precision=cg.PREC_FP32_DF_REFINE))
        got = x.cpu().numpy()
        want = np.repeat(ref[i:i + 64, None], n, axis=1)
        zero = want == 0.0   # (a smoothing may return the other zero)
        assert np.array_equal(got[zero], want[zero])
        assert np.array_equal(got.view(np.int64)[~zero], want.view(np.int64)[~zero])
    mesh.close()
