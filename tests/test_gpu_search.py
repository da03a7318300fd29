"""The radius search over the dense cell index at the sizes of its candidate
lists: from a few points around a query to several passes of 128, with the cell
box's faces within reach.  Colour off, so the costs are bit-exact against the
oracle (both J_o readings)."""
import numpy as np
import pytest

from paper_2008_00326_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jo_mode", [0, 1])
@pytest.mark.parametrize("delta,stride", [(0.003, 3), (0.004, 1), (0.008, 1), (0.016, 1), (0.03, 2), (0.06, 1), (0.3, 2)])
def test_candidate_list_sizes(oracle, delta, stride, jo_mode):
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    sc = scenes.tabletop_small()
    req = sc.requests[0]
    poses = req.poses[np.random.default_rng(5).choice(len(req.poses), 24, replace=False)]
    poses = np.concatenate([poses, req.poses[req.gt_index][None]])
    over = dict(delta_m=delta, stride=stride, jo_mode=jo_mode, color_check=0)
    with P.Context(0) as ctx:
        sid = ctx.set_observation(sc, **over)
        mid = ctx.load_mesh(sc.meshes[0])
        got = ctx.score(sid, mid, req.label, req.roi, poses)
    over["delta"] = over.pop("delta_m")
    want, _ = oracle.score(oracle.OracleScene.from_scene(sc, **over), oracle.OracleMesh.from_mesh(sc.meshes[0]),
                           poses, label=req.label, roi=req.roi)
    assert np.array_equal(got, want)


def test_few_and_many_hypotheses_score_alike():
    """Runs of up to two hypotheses per SM take larger blocks: the costs are the
    same on both sides of the line, from one hypothesis up, and under a shape the
    caller chose."""
    import torch
    from paper_2008_00326_gb300 import build, perch as P
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sc = scenes.tabletop_small(colour=True)
    req = sc.requests[0]
    with P.Context(0) as ctx:
        sid, mid = ctx.set_observation(sc), ctx.load_mesh(sc.meshes[0])
        every = ctx.score(sid, mid, req.label, req.roi, req.poses)
        assert len(every) > 2 * sms + 1
        for n in (1, 2, sms, sms + 1, 2 * sms, 2 * sms + 1):
            assert np.array_equal(ctx.score(sid, mid, req.label, req.roi, req.poses[:n]), every[:n]), n
        ctx.set_launch_config(128, 2048)
        for n in (3, 2 * sms + 1):
            assert np.array_equal(ctx.score(sid, mid, req.label, req.roi, req.poses[:n]), every[:n]), n
