"""GICP refinement at source clouds around a warp's and a block's size (a handful
of points, 31 to 33, 255 to 257, more than one pass), by restricting the render to
small regions; bit-exact against the oracle, whatever ends the iteration."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(2, 3), (5, 6), (8, 4), (11, 3), (15, 17), (16, 16), (257, 1), (40, 30)])
def test_source_cloud_sizes(oracle, size):
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    sc = scenes.tabletop_3obj(W=320, H=240, grid_half=0, tri_scale=0.2)
    rng = np.random.default_rng(9)
    gt = np.asarray(sc.gt_poses[1]).reshape(3, 4)
    u = int(round(sc.fx * gt[0, 3] / gt[2, 3] + sc.cx))
    v = int(round(sc.fy * (gt[1, 3] - 0.05) / gt[2, 3] + sc.cy))
    roi = (u - size[0] // 2, v - size[1] // 2, u - size[0] // 2 + size[0], v - size[1] // 2 + size[1])
    poses = np.tile(gt.reshape(1, 12), (6, 1))
    poses[:, [3, 7, 11]] += rng.normal(size=(6, 3)) * 0.003
    poses = poses.astype(np.float32)
    with P.Context(0) as ctx:
        sid, mid = ctx.set_observation(sc), ctx.load_mesh(sc.meshes[1])
        got, info = ctx.refine(sid, mid, -1, roi, poses)
    want, winfo = oracle.gicp(oracle.OracleScene.from_scene(sc), oracle.OracleMesh.from_mesh(sc.meshes[1]), poses,
                              label=-1, roi=roi)
    assert np.array_equal(info, winfo)
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
