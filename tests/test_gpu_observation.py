"""The observation build at its edges, through the costs it decides (bit-exact
against the oracle, colour off): a single observed pixel in a corner, none, thin
images, strides up to past the image, a cell box on both sides of the dense
index's limit; and its kept scratch, which is given back when an allocation needs
the room."""
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


def _check(P, oracle, depth, delta, stride, jo_mode=0):
    H, W = depth.shape
    f, cx, cy = 150.0, W / 2.0, H / 2.0
    mesh = scenes.box_mesh(0.2, 0.2, 0.2, 6, 6, 6)
    rng = np.random.default_rng(8)
    poses = []
    for _ in range(6):
        r = scenes.random_rotation(rng)
        poses.append(np.concatenate([r, (rng.normal(size=3) * 0.05 + [0, 0, 0.6])[:, None]], 1).reshape(12))
    poses = np.asarray(poses, np.float32)
    rgb = np.zeros((H, W, 3), np.uint8)
    params = P.perch_default_params(delta_m=delta, color_check=0, stride=stride, jo_mode=jo_mode)
    with P.Context(0) as ctx:
        mid = ctx.load_mesh(mesh)
        for _ in range(2):                      # the second build reuses the first one's scratch
            sid = P.perch_set_observation(ctx.ctx, depth, rgb, None, f, f, cx, cy, params)
            got = ctx.score(sid, mid, -1, None, poses)
            P.perch_release_scene(ctx.ctx, sid)
    osc = oracle.OracleScene(depth, rgb, None, f, f, cx, cy, delta=delta, color_check=0, stride=stride, jo_mode=jo_mode)
    want, _ = oracle.score(osc, oracle.OracleMesh.from_mesh(mesh), poses)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("shape", [(60, 80), (1, 97), (83, 1), (33, 31)])
@pytest.mark.parametrize("stride", [1, 2, 7, 500])
def test_shapes_and_strides(P, oracle, shape, stride):
    rng = np.random.default_rng(1)
    depth = rng.integers(5200, 6600, shape).astype(np.uint16)
    depth[rng.random(shape) < 0.2] = 0
    _check(P, oracle, depth, 0.01, stride)


@pytest.mark.parametrize("pixel", [None, (0, 0), (0, 79), (59, 0), (59, 79), (30, 40)])
def test_one_point_or_none(P, oracle, pixel):
    depth = np.zeros((60, 80), np.uint16)
    if pixel:
        depth[pixel] = 5500
    _check(P, oracle, depth, 0.02, 1)


@pytest.mark.parametrize("far", [6000, 30000, 65535])
@pytest.mark.parametrize("delta", [0.002, 0.005])
def test_cell_boxes_around_the_dense_limit(P, oracle, far, delta):
    rng = np.random.default_rng(2)
    depth = rng.integers(5200, 6600, (60, 80)).astype(np.uint16)
    depth[::7, ::5] = far
    for jo_mode in (0, 1):
        _check(P, oracle, depth, delta, 1, jo_mode)


def test_scratch_is_given_back(P):
    sc = scenes.tabletop_3obj(grid_half=0)
    with P.Context(0) as free:
        before = free.hbm_used
        free.set_observation(sc)
        once = free.hbm_used - before            # one scene and the scratch
    with P.Context(0, hbm_budget_bytes=before + once + 4096) as ctx:
        sids = [ctx.set_observation(sc)]
        P.perch_release_scene(ctx.ctx, sids.pop())
        sids.append(ctx.set_observation(sc))     # the scratch is still there, or its room is
        # a second scene needs the scratch's room; what cannot fit is refused and leaves nothing behind
        used = ctx.hbm_used
        with pytest.raises(P.PerchError) as e:
            for _ in range(8):
                sids.append(ctx.set_observation(sc))
        assert e.value.status == -3 and ctx.hbm_used <= before + once + 4096
        for s in sids:
            P.perch_release_scene(ctx.ctx, s)
        assert ctx.hbm_used <= used
        ctx.set_observation(sc)


def test_kept_scratch_leaves_the_hash_its_room(P):
    rng = np.random.default_rng(2)
    depth = rng.integers(5200, 6600, (60, 80)).astype(np.uint16)
    depth[::7, ::5] = 30000
    rgb = np.zeros((60, 80, 3), np.uint8)

    def build(ctx, delta):
        return P.perch_set_observation(ctx.ctx, depth, rgb, None, 150.0, 150.0, 40.0, 30.0,
                                       P.perch_default_params(delta_m=delta, color_check=0))

    def fits(budget):
        try:
            with P.Context(0, hbm_budget_bytes=budget) as ctx:
                build(ctx, 0.005)               # some 38 million cells: the hash
            return True
        except P.PerchError as e:
            assert e.status == -3
            return False

    lo, hi = 1 << 20, 64 << 20
    assert fits(hi)
    while hi - lo > 32 << 10:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid) else (mid, hi)
    with P.Context(0, hbm_budget_bytes=hi) as ctx:
        sid = build(ctx, 0.018)                 # some 0.8 million cells: 3.3 MB of scratch stay
        P.perch_release_scene(ctx.ctx, sid)
        build(ctx, 0.005)
