"""Regions of interest that end at, cross or lie past each edge of the image, and
objects that project far outside it (an empty render box either way): costs
bit-exact against the oracle, by label and by cylinder, in both J_o readings."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu

W, H = 160, 120
ROIS = [(W - 1, 0, W + 40, H), (W, 0, W + 40, H), (W + 1, 3, W + 2, 5), (0, H - 1, W, H + 1), (0, H, W, H + 9),
        (-30, -30, 0, 0), (-30, -30, 1, 1), (W + 5, H + 5, W + 50, H + 50), (5, H + 7, 60, H + 7),
        (0, 64512, W, 64600), (64512, 64512, 70000, 70000), (67108867, 0, 67108900, H), (2 ** 31 - 1,) * 4]


@pytest.mark.parametrize("jo_mode", [0, 1])
@pytest.mark.parametrize("stride", [1, 3])
def test_regions_past_the_edges(oracle, jo_mode, stride):
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    sc = scenes.sixdof_5obj(W=W, H=H, n_hyp=6, tri_scale=0.05)
    over = dict(stride=stride, jo_mode=jo_mode, color_check=0)
    osc = oracle.OracleScene.from_scene(sc, **over)
    with P.Context(0) as ctx:
        sid = ctx.set_observation(sc, **over)
        req = sc.requests[0]
        mid, om = ctx.load_mesh(sc.meshes[0]), oracle.OracleMesh.from_mesh(sc.meshes[0])
        out = np.repeat(np.asarray(sc.gt_poses[0], np.float32).reshape(1, 12), 4, 0)
        for pose, u, v in zip(out, (0, 0, 64512, -64512), (64512, 200000, 0, 0)):
            pose[11] = 0.3
            pose[3], pose[7] = (u - sc.cx) / sc.fx * 0.3, (v - sc.cy) / sc.fy * 0.3
        poses = np.concatenate([req.poses, out])
        for label in (-1, req.label):
            for roi in [None] + ROIS:
                got = ctx.score(sid, mid, label, roi, poses)
                want, _ = oracle.score(osc, om, poses, label=label, roi=roi)
                assert np.array_equal(got, want), (label, roi)
