"""Which launch shape a run takes when nobody chose one, seen by the vertex caches
that it allocates (one per resident block), and that every shape gives the same
costs."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu

FEW, BASE = (512, 14336), (256, 7064)


@pytest.fixture(scope="module")
def P():
    from paper_2008_00326_gb300 import build, perch
    build.build()
    perch.load()
    return perch


def _run(P, n, shape=None, **over):
    """(costs, bytes of scratch) of the first run of a new context."""
    import torch
    sc = scenes.tabletop_small()
    req = sc.requests[0]
    poses = torch.from_numpy(np.resize(req.poses, (n, 12))).cuda()
    costs = torch.zeros((n, 2), dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with P.Context(0) as ctx:
        sid, mid = ctx.set_observation(sc, **over), ctx.load_mesh(sc.meshes[0])
        if shape:
            ctx.set_launch_config(*shape)
        before = ctx.hbm_used
        ctx.score(sid, mid, req.label, req.roi, poses, costs, stream=stream)
        used = ctx.hbm_used - before
        P.perch_sync(ctx.ctx, stream)
    return costs.cpu().numpy(), used


@pytest.mark.parametrize("jo_mode", [0, 1])
def test_short_runs_end_at_half_the_sms(P, jo_mode):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, sms // 2, sms // 2 + 1, sms, 2 * sms, 2 * sms + 1):
        costs, used = _run(P, n, jo_mode=jo_mode)
        few, base = _run(P, n, FEW, jo_mode=jo_mode), _run(P, n, BASE, jo_mode=jo_mode)
        assert few[1] != base[1]
        assert used == (few if 2 * n <= sms else base)[1], n
        assert np.array_equal(costs, few[0]) and np.array_equal(costs, base[0]), n


def test_short_runs_on_wide_images(P, oracle):
    """Eq. 3's keys of one image row leave room for the scratch of eight warps, not of
    sixteen: a run of a few poses takes the shape of a longer one."""
    H, W, f = 4, 23000, 100.0
    rng = np.random.default_rng(3)
    depth = rng.integers(5850, 6050, (H, W)).astype(np.uint16)
    rgb = np.zeros((H, W, 3), np.uint8)
    mesh = scenes.box_mesh(0.3, 0.015, 0.015, 30, 3, 3)
    pose = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0.59], np.float32)
    step = np.float32(0.05) * (np.arange(12) == 3) - np.float32(0.02) * (np.arange(12) == 11)
    poses = np.stack([pose + k * step for k in range(3)]).astype(np.float32)
    over = dict(color_check=0, stride=1, jo_mode=1)
    with P.Context(0) as ctx:
        mid = ctx.load_mesh(mesh)
        sid = P.perch_set_observation(ctx.ctx, depth, rgb, None, f, f, W / 2.0, H / 2.0,
                                      P.perch_default_params(delta_m=0.01, **over))
        got = ctx.score(sid, mid, -1, None, poses)
    osc = oracle.OracleScene(depth, rgb, None, f, f, W / 2.0, H / 2.0, delta=0.01, **over)
    want, _ = oracle.score(osc, oracle.OracleMesh.from_mesh(mesh), poses)
    assert want[:, 1].max() > want[:, 1].min() and np.array_equal(got, want)
