"""The sorted copy of a mesh's vertices that ADD-S reads: made by the first call that
uses it, charged to the budget then, and given back when the budget needs its room; a
captured call does without it."""
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


def pairs(n, seed=4):
    rng = np.random.default_rng(seed)
    true = np.empty((n, 3, 4))
    true[:, :, :3] = scenes.rodrigues_batch(rng.normal(size=(n, 3)), rng.uniform(0, 3, n))
    true[:, :, 3] = rng.normal(size=(n, 3)) * 0.1 + [0, 0, 0.9]
    est = true.copy()
    est[:, :, :3] = scenes.rodrigues_batch(rng.normal(size=(n, 3)), rng.normal(size=n) * 0.2) @ est[:, :, :3]
    est[:, :, 3] += rng.normal(size=(n, 3)) * 0.01
    return est.reshape(n, 12).astype(np.float32), true.reshape(n, 12).astype(np.float32)


MESH = scenes.ellipsoid_mesh(0.04, 0.03, 0.05, 41, 40)


def test_made_by_the_first_call_that_uses_it(P):
    est, true = pairs(5)
    nv, nt = len(MESH.verts), len(MESH.tris)
    with P.Context(0) as ctx:
        before = ctx.hbm_used
        mid = ctx.load_mesh(MESH)
        assert ctx.hbm_used == before + 16 * (nv + nt)      # vertices and triangles, nothing else
        P.perch_add_s(ctx.ctx, mid, est, true, False)
        used = ctx.hbm_used
        P.perch_add_s(ctx.ctx, mid, est, true, True)
        assert ctx.hbm_used == used + 16 * 33 * -(-nv // 32)
        P.perch_add_s(ctx.ctx, mid, est, true, True)
        assert ctx.hbm_used == used + 16 * 33 * -(-nv // 32)
        P.perch_release_mesh(ctx.ctx, mid)
        assert ctx.hbm_used == used - 16 * (nv + nt)


def test_captured_calls(P):
    import torch
    est, true = pairs(7)
    dev = [torch.from_numpy(x).cuda() for x in (est, true)]
    out = torch.zeros(7, dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with P.Context(0) as ctx:
        mid = ctx.load_mesh(MESH)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            P.perch_add_s(ctx.ctx, mid, *dev, True, out=out, stream=stream)
        for _ in range(2):                                  # before and after the copy exists
            graph.replay()
            torch.cuda.synchronize()
            got = out.cpu().numpy()
            np.testing.assert_allclose(got, P.perch_add_s(ctx.ctx, mid, est, true, True), rtol=1e-13)
            out.zero_()
        del graph


def test_given_back_when_the_budget_needs_its_room(P):
    """The smallest budget that a program manages with when it asks for ADD is enough
    when it asks for ADD-S."""
    mesh = scenes.ellipsoid_mesh(0.04, 0.03, 0.05, 21, 20)      # 8 KB of groups
    est, true = pairs(5)
    sc = scenes.tabletop_3obj(grid_half=0)

    def program(budget, symmetric):
        with P.Context(0, hbm_budget_bytes=budget) as ctx:
            mid = ctx.load_mesh(mesh)
            first = P.perch_add_s(ctx.ctx, mid, est, true, symmetric)
            ctx.set_observation(sc)
            again = P.perch_add_s(ctx.ctx, mid, est, true, symmetric)
            assert ctx.hbm_used <= budget
            return first, again

    def fits(budget, symmetric):
        try:
            program(budget, symmetric)
            return True
        except P.PerchError as e:
            assert e.status == -3
            return False

    lo, hi = 1 << 20, 64 << 20
    assert fits(hi, False)
    while hi - lo > 1 << 10:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid, False) else (mid, hi)
    assert fits(hi, True)
    want = program(64 << 20, True)[0]
    for got in program(hi, True):
        np.testing.assert_allclose(got, want, rtol=1e-13)
