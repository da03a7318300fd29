"""ADD-S over sorted vertex groups against all pairs, in the same binary32
arithmetic (numpy, one operation at a time): vertex counts around a group's 32,
poses that coincide, lie far apart, stretch or mirror the mesh, and few and many
pairs (one or several blocks each).  The minima are the same numbers, so the means
differ by their binary64 summation order alone."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu


def _xform(P, v):
    P = P.reshape(3, 4)
    return np.stack([((P[i, 0] * v[:, 0] + P[i, 1] * v[:, 1]) + P[i, 2] * v[:, 2]) + P[i, 3] for i in range(3)], 1)


def _all_pairs(v, a, b):
    x, y = _xform(a, v), _xform(b, v)
    best = np.full(len(x), np.float32(3e38))
    for j in range(0, len(y), 256):
        d = x[:, None] - y[None, j:j + 256]
        best = np.minimum(best, ((d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]).min(1))
    return np.sqrt(best.astype(np.float64)).mean()


def _pairs(rng, n):
    true = np.empty((n, 3, 4))
    true[:, :, :3] = scenes.rodrigues_batch(rng.normal(size=(n, 3)), rng.uniform(0, 3, n))
    true[:, :, 3] = rng.normal(size=(n, 3)) * 0.1 + [0, 0, 0.9]
    est = true.copy()
    est[:, :, :3] = scenes.rodrigues_batch(rng.normal(size=(n, 3)), rng.normal(size=n) * 0.2) @ est[:, :, :3]
    est[:, :, 3] += rng.normal(size=(n, 3)) * 0.01
    est[0] = true[0]                                         # the same pose
    if n > 4:
        est[1, :, 3] += 2.0                                  # far apart
        est[2, :, :3] *= np.array([0.2, 1.7, 3.0])           # stretched
        true[3, :, 0] *= -1                                  # mirrored
        est[4, :, :3] = 0.0                                  # a point
    return est.reshape(n, 12).astype(np.float32), true.reshape(n, 12).astype(np.float32)


@pytest.mark.parametrize("verts,n", [(1, 5), (2, 1), (31, 5), (32, 5), (33, 7), (65, 3000), (500, 300), (1024, 9), (3001, 6)])
def test_groups_equal_all_pairs(verts, n):
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    rng = np.random.default_rng(verts)
    v = (rng.normal(size=(verts, 3)) * [0.03, 0.05, 0.02]).astype(np.float32)
    if verts > 300:
        v[:, 2] = np.abs(v[:, 2])
        v[verts // 2:, 0] = 0.01                             # a flat part
    mesh = scenes.Mesh("points", v, np.zeros((verts, 3), np.uint8), np.zeros((1, 3), np.int32), 0.01, 0.01)
    est, true = _pairs(rng, n)
    with P.Context(0) as ctx:
        got = P.perch_add_s(ctx.ctx, ctx.load_mesh(mesh), est, true, True)
    pick = range(n) if n < 400 else list(range(8)) + list(rng.integers(0, n, 40))
    want = np.array([_all_pairs(v, est[i], true[i]) for i in pick])
    np.testing.assert_allclose(got[list(pick)], want, rtol=1e-13, atol=1e-18)
