"""ADD-S of one pose pair: the same bits whatever other pairs share the call (their
number decides how many blocks a pair gets), below and above the number of groups
that shared memory holds, against the kernel over all pairs (a context whose budget
has no room for the sorted vertices) and against binary64 nearest neighbours."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2008_00326_gb300 import build, perch
    build.build()
    perch.load()
    return perch


def _pairs(n, seed):
    rng = np.random.default_rng(seed)
    true = np.empty((n, 3, 4))
    true[:, :, :3] = scenes.rodrigues_batch(rng.normal(size=(n, 3)), rng.uniform(0, 3, n))
    true[:, :, 3] = rng.normal(size=(n, 3)) * 0.1 + [0, 0, 0.9]
    est = true.copy()
    est[:, :, :3] = scenes.rodrigues_batch(rng.normal(size=(n, 3)), rng.normal(size=n) * 0.2) @ est[:, :, :3]
    est[:, :, 3] += rng.normal(size=(n, 3)) * 0.01
    return est.reshape(n, 12).astype(np.float32), true.reshape(n, 12).astype(np.float32)


def _points(verts):
    rng = np.random.default_rng(verts)
    v = (rng.normal(size=(verts, 3)) * [0.03, 0.05, 0.02]).astype(np.float32)
    return scenes.Mesh("points", v, np.zeros((verts, 3), np.uint8), np.zeros((1, 3), np.int32), 0.01, 0.01)


@pytest.mark.parametrize("verts", [20, 500, 1024, 3001, 33000])
def test_a_pair_alone_and_among_others(P, verts):
    est, true = _pairs(3000 if verts < 10000 else 1300, 1)
    with P.Context(0) as ctx:
        mid = ctx.load_mesh(_points(verts))
        every = P.perch_add_s(ctx.ctx, mid, est, true, True)
        for n in (1, 3, 310, 700, 1250):
            assert np.array_equal(P.perch_add_s(ctx.ctx, mid, est[:n], true[:n], True), every[:n]), n


@pytest.mark.parametrize("verts", [3001, 32768, 32769, 41000])
def test_groups_against_all_pairs(P, verts):
    from scipy.spatial import cKDTree
    mesh = _points(verts)
    est, true = _pairs(6, 2)
    with P.Context(0) as ctx:
        base = ctx.hbm_used
        mid = ctx.load_mesh(mesh)
        got = P.perch_add_s(ctx.ctx, mid, est, true, True)
        used = ctx.hbm_used - 16 * 33 * -(-verts // 32)     # without the groups
    with P.Context(0, hbm_budget_bytes=used + 64) as ctx:
        assert ctx.hbm_used == base
        every = P.perch_add_s(ctx.ctx, ctx.load_mesh(mesh), est, true, True)
        assert ctx.hbm_used == used
    # the same minima, summed in another order
    np.testing.assert_allclose(got, every, rtol=1e-13)
    for i in range(len(est)):
        a, b = (x[i].astype(np.float64).reshape(3, 4) for x in (est, true))
        v = mesh.verts.astype(np.float64)
        want = cKDTree(v @ b[:, :3].T + b[:, 3]).query(v @ a[:, :3].T + a[:, 3])[0].mean()
        assert abs(got[i] - want) < 2e-6
